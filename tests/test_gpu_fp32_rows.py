"""The persistent fp32 solve: row blocks with more rows than a block has threads (H = 8 runs on 32), several row blocks per cluster,
and the sizes around which the coarsest level of the forward solve goes to the chain kernel.  Forward, adjoint and gradients against the fp64 oracle at the same
cycle count."""
import numpy as np
import pytest

from oracle import mgrit_gru_oracle as O
from paper_2203_04738_b200.synthetic import Workload, make_inputs
from tests.gpu_util import oracle_params, to_dev, upload

pytestmark = pytest.mark.gpu


def norm(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)


def solve_against_the_oracle(T, B, H, cf, L, rf, rc, iters):
    from paper_2203_04738_b200 import binding as Bd
    ragged = T % cf ** (L - 1) != 0
    w = Workload("rows", T=T, B=B, I=16, H=H, cf=cf, levels=L, iters_fwd=iters, iters_adj=iters, relax_fine=rf, relax_coarse=rc,
                 operands=0, classes=4, relu=False, seed=T + H)
    d = make_inputs(w)
    d["h0"] = (np.random.default_rng(1).standard_normal(d["h0"].shape) * 0.3).astype(np.float32)
    p, x, h0 = upload(d)
    P = oracle_params(d)
    kw = dict(cf=cf, levels=L, relax_fine=rf, relax_coarse=rc)
    cfg = Bd.make_cfg(T, B, 16, H, iters=iters, operands=0, flags=Bd.FLAG_RAGGED_T if ragged else 0, **kw)
    xr, h0r = d["x"].astype(np.float64), d["h0"].astype(np.float64)
    seed = np.random.default_rng(2).standard_normal((T, B, H)).astype(np.float32)
    h, gi, rn = Bd.mgrit_gru_forward(cfg, p, x, h0, want_resnorm=L > 1)
    r = Bd.mgrit_gru_adjoint(cfg, p, x, h0, gi, h, dh_seed=to_dev(seed))
    assert Bd.last_device_status() == 0
    href, rref = O.mgrit_forward(*P, xr, h0r, iters=iters, ragged=ragged, **kw)      # (one level: the serial sweep)
    # 2^-24 per operation through at most T dependent steps of a contraction; the gates keep the factor near one
    assert norm(h.cpu().numpy(), href) < 5e-6
    assert L == 1 or np.allclose(rn, rref, rtol=1e-3, atol=1e-5 * rref[0] + 1e-6)
    lam, lam0, g, _ = O.mgrit_adjoint(*P, xr, h0r, h.cpu().numpy().astype(np.float64), seed.astype(np.float64), iters=iters, ragged=ragged, **kw)
    assert norm(r.dh.cpu().numpy(), lam) < 5e-6 and norm(r.dh0.cpu().numpy(), lam0) < 2e-5
    # (sums of T*B terms of either sign: 2^-24 of the running sum per addition, over at most some thousand additions a range)
    for k in ("dx", "dW_ih", "dW_hh", "db_ih", "db_hh"):
        assert norm(getattr(r, k).cpu().numpy(), g[k]) < 1e-5, k


#        T    B    H   cf L  rf rc iters     rows of the largest phase: 6500 and 12800, blocks of 44 rows and more
MORE_ROWS_THAN_THREADS = [(258, 100, 8, 4, 2, 0, 1, 2), (512, 100, 8, 4, 3, 1, 1, 1), (1024, 32, 8, 4, 2, 0, 1, 2), (258, 100, 16, 4, 2, 1, 0, 2)]


@pytest.mark.parametrize("c", MORE_ROWS_THAN_THREADS, ids=lambda c: "T{}B{}H{}cf{}L{}r{}{}i{}".format(*c))
def test_blocks_with_more_rows_than_threads(c):
    solve_against_the_oracle(*c)


# the chain serves H = 192 and H > 256 while eight units a CTA fit one wave, and 120 rows and more at H > 192 on sixteen; inside a
# solve from 25 us on (32 steps at H > 256, 167 at H = 192): both sides of each line
CHAIN_OR_PHASE = [(7, 64, 192, 2, 1, 0, 0, 1), (7, 100, 192, 2, 1, 0, 0, 1), (9, 17, 288, 2, 1, 0, 0, 1), (5, 65, 352, 2, 1, 0, 0, 1), (6, 128, 224, 2, 1, 0, 0, 1),
                  (6, 113, 256, 2, 1, 0, 0, 1), (33, 3, 264, 2, 1, 0, 0, 1), (66, 3, 320, 2, 2, 0, 1, 2), (62, 33, 288, 2, 2, 1, 1, 2),
                  (340, 2, 192, 2, 2, 0, 1, 2), (260, 5, 352, 4, 2, 2, 1, 2)]


@pytest.mark.parametrize("c", CHAIN_OR_PHASE, ids=lambda c: "T{}B{}H{}cf{}L{}r{}{}i{}".format(*c))
def test_coarsest_level_on_the_chain_or_as_a_phase(c):
    solve_against_the_oracle(*c)


# more rows than one wave of row blocks holds, for every size of cluster (148, 74, some 35 and some 16 of them with up to 64 rows each; H = 96
# and above 256 fewer): clusters take a second and a third block, whose buffers their peers have to be done with
SEVERAL_BLOCKS = [(1024, 48, 32, 4, 2, 0, 1, 1), (512, 64, 96, 4, 2, 1, 0, 1), (515, 44, 104, 4, 2, 1, 1, 1), (259, 50, 136, 4, 3, 0, 1, 2),
                  (256, 50, 192, 4, 2, 1, 0, 1), (131, 50, 224, 4, 2, 1, 1, 1), (128, 50, 256, 4, 2, 0, 1, 1), (128, 50, 288, 4, 2, 1, 0, 1), (130, 30, 352, 4, 2, 0, 1, 1)]


@pytest.mark.parametrize("c", SEVERAL_BLOCKS, ids=lambda c: "T{}B{}H{}cf{}L{}r{}{}i{}".format(*c))
def test_clusters_with_several_row_blocks(c):
    solve_against_the_oracle(*c)
