"""The fp32 engine's gradient pass and projection at the edges of their 64 x 64 tiles and of the ranges the reduction over
T*B rows is cut into: one row, fewer rows than a tile, rows that end inside a step of sixteen, one range and many."""
import numpy as np
import pytest
import torch

from oracle import mgrit_gru_oracle as O
from paper_2203_04738_b200.synthetic import Workload, make_inputs
from tests.gpu_util import oracle_params, to_dev, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,B,I,H", [(1, 1, 8, 8), (5, 3, 72, 40), (67, 2, 8, 64), (40, 33, 136, 72), (300, 9, 16, 104)])
def test_serial_gradients_against_fp64(T, B, I, H):
    from paper_2203_04738_b200 import binding as Bd
    w = Workload("g", T=T, B=B, I=I, H=H, cf=2, levels=1, iters_fwd=1, iters_adj=1, relax_fine=0, relax_coarse=0, operands=0,
                 classes=4, relu=False, seed=T + H)
    d = make_inputs(w)
    p, x, h0 = upload(d)
    cfg = Bd.make_cfg(T, B, I, H, cf=2, levels=1, operands=0)
    h, gi = Bd.gru_serial_forward(cfg, p, x, h0)
    seed = np.random.default_rng(7).standard_normal((T, B, H)).astype(np.float32)
    r = Bd.gru_serial_backward(cfg, p, x, h0, gi, h, dh_seed=to_dev(seed))
    P = oracle_params(d)
    gi_ref = d["x"].astype(np.float64) @ P[0].T + P[2]
    norm = lambda a, b: np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)
    assert norm(gi.cpu().numpy(), gi_ref) < 1e-6
    lam, lam0, g = O.serial_backward(*P, d["x"].astype(np.float64), d["h0"].astype(np.float64), h.cpu().numpy().astype(np.float64),
                                     seed.astype(np.float64))
    # 2^-24 per operation; the sensitivities carry a chain of up to 300 steps, the reductions up to 2700 terms
    for k in ("dx", "dW_ih", "dW_hh", "db_ih", "db_hh"):
        assert norm(getattr(r, k).cpu().numpy(), g[k]) < 5e-6, k
