"""A NaN in one row of a bias reaches every state and sensitivity that depends on it, gate by gate, in every engine: the NaN
patterns are those of the oracle's serial sweep and back-propagation (a diverged run must not pass for a sound one)."""
import numpy as np
import pytest

from oracle import mgrit_gru_oracle as O
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu
NAMES = ("W_ih", "W_hh", "b_ih", "b_hh")


def inputs(gates, H, T=3, B=8, I=16):
    rng = np.random.default_rng(gates + H)
    P = [(0.2 * rng.standard_normal(s)).astype(np.float32) for s in ((gates * H, I), (gates * H, H), (gates * H,), (gates * H,))]
    return P, rng.standard_normal((T, B, I)).astype(np.float32), rng


# operands 0 and 1: up to H = 352 the persistent fp32 solve, above it the step and chain kernels (0) or the split's tiles (1)
@pytest.mark.parametrize("operands,H", [(0, 40), (0, 384), (1, 64), (1, 384), (2, 64)])
@pytest.mark.parametrize("cell", [O.CELL_CLASSIC, O.CELL_IMPLICIT])
@pytest.mark.parametrize("gate", [0, 1, 2])
def test_gru_gate(operands, H, cell, gate):
    from paper_2203_04738_b200 import binding as Bd
    P, x, rng = inputs(3, H)
    P[3][gate * H + 5] = np.nan
    T, B, I = x.shape
    h0, hlin, seed = (rng.standard_normal(s).astype(np.float32) for s in ((B, H), (T, B, H), (T, B, H)))
    p = {k: to_dev(v) for k, v in zip(NAMES, P)}
    cfg = Bd.make_cfg(T, B, I, H, operands=operands, levels=1, cell=cell)
    h, gi = Bd.gru_serial_forward(cfg, p, to_dev(x), to_dev(h0))
    P64 = [a.astype(np.float64) for a in P]
    assert np.array_equal(np.isnan(h.cpu().numpy()), np.isnan(O.serial_forward(*P64, x, h0, cell=cell)))
    r = Bd.gru_serial_backward(cfg, p, to_dev(x), to_dev(h0), gi, to_dev(hlin), dh_seed=to_dev(seed))
    lam, _, g = O.serial_backward(*P64, x, h0, hlin.astype(np.float64), seed.astype(np.float64), cell=cell)
    assert np.array_equal(np.isnan(r.dh.cpu().numpy()), np.isnan(lam))
    assert np.array_equal(np.isnan(r.db_hh.cpu().numpy()), np.isnan(g["db_hh"]))


@pytest.mark.parametrize("operands,H", [(0, 40), (1, 64), (2, 64)])
@pytest.mark.parametrize("gate", [0, 1, 2, 3])
def test_lstm_gate(operands, H, gate):
    from paper_2203_04738_b200 import binding as Bd
    P, x, rng = inputs(4, H)
    P[3][gate * H + 5] = np.nan
    T, B, I = x.shape
    u0, ulin, seed = (rng.standard_normal(s).astype(np.float32) for s in ((2, B, H), (T, 2, B, H), (T, 2, B, H)))
    p = {k: to_dev(v) for k, v in zip(NAMES, P)}
    cfg = Bd.make_cfg(T, B, I, H, operands=operands, levels=1)
    u, gi, _ = Bd.mgrit_lstm_forward(cfg, p, to_dev(x), to_dev(u0))
    P64 = [a.astype(np.float64) for a in P]
    assert np.array_equal(np.isnan(u.cpu().numpy()), np.isnan(O.lstm_serial_forward(*P64, x, u0)))
    _, _, r, _ = Bd.mgrit_lstm_adjoint(cfg, p, to_dev(x), to_dev(u0), gi, to_dev(ulin), du_seed=to_dev(seed))
    g = O.lstm_serial_backward(*P64, x, u0, ulin.astype(np.float64), seed.astype(np.float64))[2]
    assert np.array_equal(np.isnan(r.db_hh.cpu().numpy()), np.isnan(g["db_hh"]))
