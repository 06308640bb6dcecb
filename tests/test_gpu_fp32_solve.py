"""The persistent fp32 solve (forward, adjoint, linearisation) at the edges of its shapes: one CTA and clusters of two, four and
eight, widths that leave the last CTA fewer units, batch sizes around a row block of four, ragged lengths, every relaxation, more
phases than one launch holds, F-cycles, the serial sweep, and the tf32 split's small solves that take the same kernels."""
import numpy as np
import pytest
import torch

from oracle import mgrit_gru_oracle as O
from paper_2203_04738_b200.synthetic import Workload, make_inputs
from tests.gpu_util import oracle_params, to_dev, upload

pytestmark = pytest.mark.gpu

#        T    B   H   cf L  rf rc iters f_cycle operands
CASES = [(64, 2, 32, 4, 2, 0, 1, 2, False, 0), (37, 1, 8, 2, 3, 1, 0, 2, False, 0), (50, 5, 104, 4, 2, 2, 1, 2, False, 0),
         (48, 100, 104, 4, 3, 0, 1, 1, False, 0), (40, 3, 136, 2, 3, 1, 1, 2, False, 0), (33, 17, 184, 4, 2, 1, 0, 2, False, 0),
         (36, 2, 248, 3, 3, 3, 2, 2, False, 0), (64, 33, 256, 4, 2, 0, 1, 2, False, 1), (30, 4, 320, 2, 2, 1, 1, 2, False, 1),
         (96, 2, 64, 2, 5, 1, 1, 4, True, 0), (29, 6, 352, 2, 1, 0, 0, 1, False, 0), (128, 16, 64, 4, 3, 1, 1, 2, False, 1),
         (26, 21, 96, 4, 2, 1, 1, 1, False, 0), (24, 40, 128, 2, 2, 1, 1, 1, False, 0), (24, 65, 168, 2, 2, 1, 1, 1, False, 0),
         (20, 70, 216, 2, 2, 0, 1, 1, False, 0)]


@pytest.mark.parametrize("c", CASES, ids=lambda c: "T{}B{}H{}cf{}L{}r{}{}i{}{}o{}".format(*c[:8], "F" if c[8] else "V", c[9]))
def test_solve_against_the_oracle(c):
    from paper_2203_04738_b200 import binding as Bd
    T, B, H, cf, L, rf, rc, iters, fcyc, op = c
    ragged = T % cf ** (L - 1) != 0
    w = Workload("f32", T=T, B=B, I=16, H=H, cf=cf, levels=L, iters_fwd=iters, iters_adj=iters, relax_fine=rf, relax_coarse=rc,
                 operands=op, classes=4, relu=False, seed=T + H)
    d = make_inputs(w)
    d["h0"] = (np.random.default_rng(1).standard_normal(d["h0"].shape) * 0.3).astype(np.float32)
    p, x, h0 = upload(d)
    P = oracle_params(d)
    flags = (Bd.FLAG_RAGGED_T if ragged else 0) | (Bd.FLAG_F_CYCLE if fcyc else 0)
    kw = dict(cf=cf, levels=L, relax_fine=rf, relax_coarse=rc)
    okw = dict(kw, iters=iters, cycle=O.CYCLE_F if fcyc else O.CYCLE_V, ragged=ragged)
    seed = np.random.default_rng(2).standard_normal((T, B, H)).astype(np.float32)
    xr, h0r = d["x"].astype(np.float64), d["h0"].astype(np.float64)
    norm = lambda a, b: np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)
    for fl in (flags, flags | Bd.FLAG_SKIP_DUPLICATE_FRELAX):
        cfg = Bd.make_cfg(T, B, 16, H, iters=iters, operands=op, flags=fl, **kw)
        n0 = Bd.kernel_launches()
        h, gi, rn = Bd.mgrit_gru_forward(cfg, p, x, h0, want_resnorm=L > 1)
        # the projection (tf32: and its operand splits, two), one launch that clears and copies, one solve per 40 phases: at most five here
        assert Bd.kernel_launches() - n0 <= 7
        r = Bd.mgrit_gru_adjoint(cfg, p, x, h0, gi, h, dh_seed=to_dev(seed), want_resnorm=L > 1)
        if L == 1:
            href = O.serial_forward(*P, xr, h0r)
        else:
            href, rref = O.mgrit_forward(*P, xr, h0r, **okw)
        # 2^-24 per operation through at most T dependent steps of a contraction; the gates keep the factor near one
        assert norm(h.cpu().numpy(), href) < 5e-6
        hn = h.cpu().numpy().astype(np.float64)
        if L == 1:
            lam, lam0, g = O.serial_backward(*P, xr, h0r, hn, seed.astype(np.float64))
        else:
            assert np.allclose(rn, rref, rtol=1e-3, atol=1e-5 * rref[0] + 1e-6)
            lam, lam0, g, _ = O.mgrit_adjoint(*P, xr, h0r, hn, seed.astype(np.float64), **okw)
        assert norm(r.dh.cpu().numpy(), lam) < 5e-6 and norm(r.dh0.cpu().numpy(), lam0) < 2e-5
        # (the tf32 split's gradient products drop the product of the two low parts: 2^-22 of every term, and the reduction cancels)
        for k in ("dx", "dW_ih", "dW_hh", "db_ih", "db_hh"):
            assert norm(getattr(r, k).cpu().numpy(), g[k]) < (6e-5 if op else 1e-5), k
    assert Bd.last_device_status() == 0


@pytest.mark.parametrize("H", [8, 112, 160])
def test_gates_at_the_ends_of_their_range(H):
    """Pre-activations from -120 to 120, where e^-x leaves the range of fp32: against the oracle in double precision."""
    from paper_2203_04738_b200 import binding as Bd
    T, B, rng = 3, 9, np.random.default_rng(H)
    W_ih, W_hh = rng.standard_normal((3 * H, 8)).astype(np.float32), (rng.standard_normal((3 * H, H)) * H ** -0.5).astype(np.float32)
    b_ih, b_hh = rng.permutation(np.linspace(-120, 120, 3 * H)).astype(np.float32), np.zeros(3 * H, np.float32)
    x, h0 = rng.standard_normal((T, B, 8)).astype(np.float32), np.zeros((B, H), np.float32)
    p = {k: to_dev(v) for k, v in dict(W_ih=W_ih, W_hh=W_hh, b_ih=b_ih, b_hh=b_hh).items()}
    h, _ = Bd.gru_serial_forward(Bd.make_cfg(T, B, 8, H, operands=0, levels=1), p, to_dev(x), to_dev(h0))
    ref = O.serial_forward(*(v.astype(np.float64) for v in (W_ih, W_hh, b_ih, b_hh, x, h0)))
    # a pre-activation a is rounded to 2^-24 |a|, at most 2^-17 for |a| < 128, and moves its gate by that times e^-|a| / (1 + e^-|a|)^2
    # or 1 - n^2, that is by at most 2^-24 max |a| sech^2 a < 2^-24; the gates' functions add a few units of 2^-24 each, T = 3 steps
    assert np.abs(h.cpu().numpy() - ref).max() < 3 * 10 * 2.0 ** -24
