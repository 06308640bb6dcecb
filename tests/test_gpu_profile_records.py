"""The profiling records of a solve count the cell evaluations of every level, whichever kernels run them (step by step at H = 384, the
persistent fp32 solve below)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,relax", [(32, 0), (104, 1), (320, 0), (384, 1)])
def test_the_records_hold_every_step(H, relax):
    from paper_2203_04738_b200 import binding as B
    T, Bz, cf = 64, 3, 4
    g = torch.Generator(device="cuda")
    g.manual_seed(H)
    k = H ** -0.5
    p = {n: (torch.rand(*s, generator=g, device="cuda") * 2 - 1) * k
         for n, s in dict(W_ih=(3 * H, 8), W_hh=(3 * H, H), b_ih=(3 * H,), b_hh=(3 * H,)).items()}
    x, h0 = torch.randn(T, Bz, 8, generator=g, device="cuda"), torch.zeros(Bz, H, device="cuda")
    cfg = B.make_cfg(T, Bz, 8, H, cf=cf, levels=2, iters=1, relax_fine=relax, operands=0)
    h, gi, _ = B.mgrit_gru_forward(cfg, p, x, h0)
    seed = torch.randn(T, Bz, H, generator=g, device="cuda")
    nc = T // cf
    # F (CF)^relax, the step that evaluates v, the coarse right-hand side, the coarsest level, the closing F-relaxation
    rows = Bz * ((T - nc) + relax * T + nc + nc + nc + (T - nc))
    B.profile_enable(True)
    try:
        B.mgrit_gru_forward(cfg, p, x, h0)
        B.mgrit_gru_adjoint(cfg, p, x, h0, gi, h, dh_seed=seed)
        rec = B.profile_read()
    finally:
        B.profile_enable(False)
    for names in (("forward_step", "forward_serial_chain"), ("adjoint_step", "adjoint_serial_chain")):
        ms, flops = (sum(rec[n][i] for n in names) for i in (0, 2))
        assert ms > 0 and flops == 6.0 * rows * H * H, (names, rec)
