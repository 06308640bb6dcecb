"""Few-row forward steps on 32-unit tiles, two k-blocks per stage, against the same steps on 64-unit tiles: the same products summed in
the same order, so the same bits.  Widths of one, two, three, five and sixteen k-blocks (the last stage may hold one), rows that fill
a tile, a part of one and more than one, with and without additive terms (the coarse levels have them)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import sys, numpy as np, torch
from paper_2203_04738_b200 import binding as B
out = {}
for H in (64, 128, 192, 320, 1024):
    for T, Bz in ((32, 1), (64, 8), (72, 32)):
        g = torch.Generator(device="cuda"); g.manual_seed(H + Bz)
        k = H ** -0.5
        p = {n: (torch.rand(*s, generator=g, device="cuda") * 2 - 1) * k for n, s in dict(W_ih=(3 * H, 32), W_hh=(3 * H, H), b_ih=(3 * H,), b_hh=(3 * H,)).items()}
        x = torch.randn(T, Bz, 32, generator=g, device="cuda"); h0 = torch.randn(Bz, H, generator=g, device="cuda") * 0.3
        cfg = B.make_cfg(T, Bz, 32, H, cf=2, levels=3, iters=2, relax_fine=1, operands=B.OPERANDS_BF16)
        out[f"{H}_{T}_{Bz}"] = B.mgrit_gru_forward(cfg, p, x, h0)[0].cpu().numpy()
assert B.last_device_status() == 0
np.savez(sys.argv[1], **out)
"""


def test_narrow_and_wide_tiles_give_the_same_bits(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    outs = []
    for flag in ("1", "0"):
        out = str(tmp_path / f"small{flag}.npz")
        env = dict(os.environ, MGRIT_GRU_CELL_SMALL=flag, PYTHONPATH=root)
        subprocess.run([sys.executable, "-c", CHILD, out], check=True, env=env, cwd=root, timeout=600)
        outs.append(np.load(out))
    for k in outs[0].files:
        assert np.array_equal(outs[0][k], outs[1][k]), k
