"""The fused bf16 kernels where their tiles are not full: batch sizes that do not divide the 128 rows of a tile (one interval per
tile, two, many), ragged lengths whose last interval takes only some of a sweep's steps, chains of widths that are odd multiples of
64, and a coarsest level whose rows do not fit the chain kernel (it runs as sweeps over one interval).  Forward, adjoint and
gradients against the fp64 oracle at the same cycle count; the sweeps must also repeat bit for bit."""
import numpy as np
import pytest
import torch

from oracle import mgrit_gru_oracle as O
from paper_2203_04738_b200.synthetic import Workload, make_inputs
from tests.gpu_util import oracle_params, rel_inf, to_dev, upload

pytestmark = pytest.mark.gpu

#        T    B    I    H   cf L  rf rc
CASES = [(64, 3, 16, 64, 4, 2, 0, 1), (61, 24, 48, 192, 4, 3, 1, 1), (50, 40, 16, 320, 2, 3, 0, 2), (48, 100, 32, 256, 4, 2, 1, 0),
         (127, 127, 16, 128, 4, 3, 0, 1), (40, 65, 16, 576, 2, 2, 1, 1), (44, 100, 64, 1024, 2, 2, 0, 1), (163, 8, 16, 64, 8, 2, 2, 0),
         (33, 128, 16, 64, 4, 2, 0, 0), (16, 130, 16, 64, 2, 2, 1, 0), (2047, 8, 16, 512, 4, 3, 1, 1)]


@pytest.mark.parametrize("c", CASES, ids=lambda c: "T{}B{}I{}H{}cf{}L{}r{}{}".format(*c))
def test_partial_tiles_against_the_oracle(c):
    from paper_2203_04738_b200 import binding as Bd
    T, B, I, H, cf, L, rf, rc = c
    if T * B % 8:
        T -= T % 8                                     # (the engine needs whole groups of eight rows)
    ragged = T % cf ** (L - 1) != 0
    w = Workload("any", T=T, B=B, I=I, H=H, cf=cf, levels=L, iters_fwd=2, iters_adj=2, relax_fine=rf, relax_coarse=rc, operands=2,
                 classes=4, relu=True, seed=T + B + H)
    d = make_inputs(w)
    d["h0"] = (np.random.default_rng(1).standard_normal(d["h0"].shape) * 0.3).astype(np.float32)
    p, x, h0 = upload(d)
    P = oracle_params(d)
    kw = dict(cf=cf, levels=L, relax_fine=rf, relax_coarse=rc)
    flags = (Bd.FLAG_RAGGED_T if ragged else 0) | Bd.FLAG_GI_CARRIES_COPIES
    cfg = Bd.make_cfg(T, B, I, H, iters=2, operands=2, flags=flags, **kw)
    h, gi, _ = Bd.mgrit_gru_forward(cfg, p, x, h0)
    for _ in range(2):
        assert torch.equal(Bd.mgrit_gru_forward(cfg, p, x, h0)[0], h)
    rows = [0, B // 2, B - 1]                          # batch rows never interact: the oracle runs a few of them
    big = T * B * H > 3e6
    xr, h0r = d["x"].astype(np.float64), d["h0"].astype(np.float64)
    if big:
        xr, h0r = xr[:, rows], h0r[rows]
    pick = lambda a: a[:, rows] if big else a
    href, _ = O.mgrit_forward(*P, xr, h0r, iters=2, ragged=ragged, **kw)
    assert rel_inf(pick(h.cpu().numpy()), href) < 2e-2
    seed = np.random.default_rng(2).standard_normal((T, B, H)).astype(np.float32)
    r = Bd.mgrit_gru_adjoint(cfg, p, x, h0, gi, h, dh_seed=to_dev(seed))
    hn = h.cpu().numpy().astype(np.float64)
    lam, lam0, g, _ = O.mgrit_adjoint(*P, xr, h0r, pick(hn), pick(seed).astype(np.float64), iters=2, ragged=ragged, **kw)
    assert rel_inf(pick(r.dh.cpu().numpy()), lam) < 2e-2 and rel_inf(r.dh0.cpu().numpy()[rows] if big else r.dh0.cpu().numpy(), lam0) < 2e-2
    assert rel_inf(pick(r.dx.cpu().numpy()), g["dx"]) < 2e-2
    if not big:
        for k in ("dW_ih", "dW_hh", "db_ih", "db_hh"):
            assert rel_inf(getattr(r, k).cpu().numpy(), g[k]) < 2e-2, k
    assert Bd.last_device_status() == 0
