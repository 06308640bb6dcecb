"""The small tf32-split shapes on the tensor cores.  Their solves go to the persistent fp32 kernels, so that the tile edges that
test_gpu_parity_tf32.py is made of (rows that straddle intervals, a partial last tile, three gate tiles) no longer meet the tf32
products there: its cases once more in a process in which those kernels are switched off (the switch is read once)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu


def test_parity_cases_on_the_tf32_products():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-m", "gpu", "-k", "not full_size", "tests/test_gpu_parity_tf32.py"],
                       env=dict(os.environ, MGRIT_GRU_F32_SOLVE="0", PYTHONPATH=root), cwd=root, timeout=900, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
