"""MGRIT_FLAG_GI_CARRIES_COPIES where B does not divide 128: ignored, as the header says.  The forward call leaves everything behind
the projection alone, and the adjoint call serves a projection that another call made and states of the caller's own."""
import numpy as np
import pytest
import torch

from paper_2203_04738_b200.synthetic import Workload, make_inputs
from tests.gpu_util import to_dev, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Bsz", [24, 100, 130])
def test_flag_is_ignored_where_the_batch_does_not_divide_a_tile(Bsz):
    from paper_2203_04738_b200 import binding as B
    w = Workload("contract", T=64, B=Bsz, I=64, H=128, cf=4, levels=2, iters_fwd=2, iters_adj=2, relax_fine=0, relax_coarse=1,
                 operands=2, classes=8, relu=True, seed=5)
    p, x, h0 = upload(make_inputs(w))
    kw = dict(cf=w.cf, levels=w.levels, iters=2, relax_fine=0, relax_coarse=1, operands=2)
    plain = B.make_cfg(w.T, Bsz, w.I, w.H, **kw)
    carry = B.make_cfg(w.T, Bsz, w.I, w.H, flags=B.FLAG_GI_CARRIES_COPIES | B.FLAG_GI_F32_UNUSED, **kw)
    n = w.T * Bsz * 3 * w.H
    # the buffers have room for copies; what is behind the projection is NaN and has to stay it
    buf = B.alloc_gi(carry, x.device).fill_(float("nan"))
    h, gi, _ = B.mgrit_gru_forward(plain, p, x, h0)
    h2, _, _ = B.mgrit_gru_forward(carry, p, x, h0, gi=buf)
    assert torch.equal(h, h2) and torch.equal(buf[:n], gi.reshape(-1)) and bool(torch.isnan(buf[n:]).all())
    buf2 = B.alloc_gi(carry, x.device).fill_(float("nan"))
    B.gru_input_projection(plain, p, x, gi=buf2[:n].view(w.T, Bsz, 3 * w.H))
    own = to_dev(np.random.default_rng(3).uniform(-0.5, 0.5, tuple(h.shape)).astype(np.float32))
    seed = to_dev(np.random.default_rng(4).standard_normal(tuple(h.shape)).astype(np.float32))
    a = B.mgrit_gru_adjoint(plain, p, x, h0, gi, own, dh_seed=seed)
    b = B.mgrit_gru_adjoint(carry, p, x, h0, buf2, own, dh_seed=seed)
    for k in ("dh", "dh0", "dx", "dW_ih", "dW_hh", "db_ih", "db_hh"):
        assert torch.equal(getattr(a, k), getattr(b, k)), k
    assert B.last_device_status() == 0
