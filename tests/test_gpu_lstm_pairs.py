"""LSTM steps and linearisation on CTA pairs (more than 128 rows) against the single-CTA kernel (up to 128): rows are independent, so a
batch that is repeated has to give every copy the states and sensitivities of the batch alone.  Row counts around a pair's 256 rows,
ragged last tiles, one and three unit tiles, every kind of update (plain, additive term, residual)."""
import numpy as np
import pytest
import torch

from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,copies,cf,cell", [(64, 3, 2, 0), (64, 17, 2, 1), (192, 5, 2, 0), (192, 4, 4, 0), (320, 33, 2, 0)])
def test_copies_of_a_batch(H, copies, cf, cell):
    from paper_2203_04738_b200 import binding as Bd
    T, B, I = 16, 8, 16
    rng = np.random.default_rng(H + copies)
    k = H ** -0.5
    p = {n: to_dev(rng.uniform(-k, k, s).astype(np.float32)) for n, s in dict(W_ih=(4 * H, I), W_hh=(4 * H, H), b_ih=(4 * H,), b_hh=(4 * H,)).items()}
    x = to_dev(rng.standard_normal((T, B, I)).astype(np.float32))
    u0 = to_dev((rng.standard_normal((2, B, H)) * 0.3).astype(np.float32))
    seed = to_dev(rng.standard_normal((T, 2, B, H)).astype(np.float32))

    def solve(n):
        cfg = Bd.make_cfg(T, B * n, I, H, cf=cf, levels=2, iters=2, cell=cell, relax_fine=1, operands=Bd.OPERANDS_BF16)
        xs, us, ds = (torch.cat([v] * n, dim=d).contiguous() for v, d in ((x, 1), (u0, 1), (seed, 2)))
        u, gi, _ = Bd.mgrit_lstm_forward(cfg, p, xs, us)
        return u, Bd.mgrit_lstm_adjoint(cfg, p, xs, us, gi, u, du_seed=ds)

    u1, (du1, du01, g1, _) = solve(1)
    un, (dun, du0n, gn, _) = solve(copies)
    rel = lambda a, b: float((a - b).norm() / b.norm())
    # A sum in another order differs by 2^-24 sqrt(H) and moves a state over a rounding boundary of its bf16 copy, 2^-8 wide, with
    # probability 2^-16 sqrt(H): 2^-8 sqrt(2^-16 sqrt(H)) = 2^-16 H^(1/4) < 7e-5 a step, 4 times that over T = 16 independent ones;
    # the adjoint's operand and its bf16 coefficients pass through the same three times
    for c in range(copies):
        s = slice(c * B, (c + 1) * B)
        assert rel(un[:, :, s], u1) < 3e-4
        assert rel(dun[:, :, s], du1) < 1e-3 and rel(du0n[:, s], du01) < 1e-3
    for n in ("dW_ih", "dW_hh", "db_ih", "db_hh"):
        assert rel(getattr(gn, n), copies * getattr(g1, n)) < 1e-3, n
    assert Bd.last_device_status() == 0
