"""A C-step inside one launch of adjoint steps replaces the rows that the next interval started from, which another group of CTAs may
not have read yet when the device is shared.  Solves with several row tiles per launch and a C-step in it, repeated while ordinary
kernels of another stream hold part of the SMs: the same bits as on an idle device, every time.  Batches that divide the tile, that do
not, and that are larger than one."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# T, batch, H, cf, levels, relax_fine: rows of the launches with a C-step (level 0 where relax_fine is 1, level 1 otherwise)
CASES = [(2048, 8, 1024, 4, 3, 0), (128, 100, 1024, 4, 3, 0), (1024, 32, 512, 4, 3, 0), (24, 136, 704, 4, 2, 1), (217, 24, 576, 4, 2, 1)]


@pytest.mark.parametrize("c", CASES, ids=lambda c: "T{}B{}H{}".format(*c))
def test_a_shared_device_changes_no_bit(c):
    from paper_2203_04738_b200 import binding as B
    T, Bz, H, cf, L, relax = c
    g = torch.Generator(device="cuda")
    g.manual_seed(H + Bz)
    k = H ** -0.5
    p = {n: (torch.rand(*s, generator=g, device="cuda") * 2 - 1) * k for n, s in dict(W_ih=(3 * H, 64), W_hh=(3 * H, H), b_ih=(3 * H,), b_hh=(3 * H,)).items()}
    x, h0, seed = torch.randn(T, Bz, 64, generator=g, device="cuda"), torch.zeros(Bz, H, device="cuda"), torch.randn(T, Bz, H, generator=g, device="cuda")
    cfg = B.make_cfg(T, Bz, 64, H, cf=cf, levels=L, iters=2, relax_fine=relax, relax_coarse=1, operands=B.OPERANDS_BF16, flags=B.FLAG_RAGGED_T if T % cf else 0)
    h, gi, _ = B.mgrit_gru_forward(cfg, p, x, h0)
    solve = lambda kw: B.mgrit_gru_adjoint(cfg, p, x, h0, gi, h, want_dx=False, **kw)
    a, b = torch.randn(2048, 2048, generator=g, device="cuda"), torch.empty(2048, 2048, device="cuda")
    small = torch.randn(40 * 4096, generator=g, device="cuda")      # (a few dozen blocks a kernel: some of the SMs)
    side = torch.cuda.Stream()
    for kw in (dict(dh_seed=seed), dict(dhT=seed[-1])):
        ref = solve(kw)
        torch.cuda.synchronize()
        for _ in range(6):
            with torch.cuda.stream(side):
                for i in range(40):
                    torch.mm(a, a, out=b)
                    small.sin_()
            r = solve(kw)
            assert torch.equal(r.dh, ref.dh) and torch.equal(r.dh0, ref.dh0) and torch.equal(r.dW_hh, ref.dW_hh)
        torch.cuda.synchronize()
    assert B.last_device_status() == 0
