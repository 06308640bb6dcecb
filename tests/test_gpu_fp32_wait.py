"""The bounded wait of the persistent fp32 solve.  Clusters without work in the coarsest level wait for its whole serial chain, here
57 ms and more: a limit of 5 ms without progress must not end that (the chain reports while it runs), and a limit shorter than the
time between two reports must: the calls return, the status tells of it, and the library works again once it is cleared.  The limit
is read once per process, so each one runs in a child process."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import sys, numpy as np, torch
from paper_2203_04738_b200 import binding as B
def solve(T, H):
    g = torch.Generator(device="cuda"); g.manual_seed(H)
    k = H ** -0.5
    p = {n: (torch.rand(*s, generator=g, device="cuda") * 2 - 1) * k for n, s in dict(W_ih=(3 * H, 8), W_hh=(3 * H, H), b_ih=(3 * H,), b_hh=(3 * H,)).items()}
    x, h0, seed = torch.randn(T, 1, 8, generator=g, device="cuda"), torch.zeros(1, H, device="cuda"), torch.randn(T, 1, H, generator=g, device="cuda")
    cfg = B.make_cfg(T, 1, 8, H, cf=2, levels=2, iters=1, relax_fine=0, operands=0)
    h, gi, _ = B.mgrit_gru_forward(cfg, p, x, h0)
    r = B.mgrit_gru_adjoint(cfg, p, x, h0, gi, h, dh_seed=seed)
    return h, r.dh
if sys.argv[2] == "long":
    h, dh = solve(1 << 17, 32)
    assert B.last_device_status() == 0
    np.savez(sys.argv[1], h=h.cpu().numpy(), dh=dh.cpu().numpy())
else:
    solve(1 << 14, 256)                    # 256 steps of 2.9 us and more between two reports
    assert B.last_device_status() == -6
    B.clear_device_status()
    assert B.last_device_status() == 0
    h, dh = solve(64, 32)                  # (no wait of this one lasts long enough for the limit to be looked at twice)
    assert B.last_device_status() == 0 and bool(torch.isfinite(h).all()) and bool(torch.isfinite(dh).all())
"""


def run(tmp_path, us, what):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = str(tmp_path / f"wait{us}.npz")
    subprocess.run([sys.executable, "-c", CHILD, out, what], check=True, env=dict(os.environ, MGRIT_GRU_TEST_F32_WAIT_US=str(us), PYTHONPATH=root),
                   cwd=root, timeout=600)
    return out


def test_a_long_chain_is_not_a_wait_without_progress(tmp_path):
    a, b = np.load(run(tmp_path, 2000000, "long")), np.load(run(tmp_path, 5000, "long"))
    for k in a.files:
        assert np.array_equal(a[k], b[k]), k


def test_a_wait_that_runs_out_is_reported(tmp_path):
    run(tmp_path, 1, "short")
