"""The loss head at the edges of its launch rules: rows that allow 16-byte loads and rows that do not (H % 4), class counts
around the four classes a warp handles at a time and around sixteen warps of them, one batch row and many, unlabelled rows."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,C", [(1, 8, 1), (3, 33, 5), (2, 104, 64), (100, 1024, 51), (16, 256, 65), (5, 4100, 130), (2, 36, 8192)])
def test_head_against_fp64(B, H, C):
    from paper_2203_04738_b200 import binding as Bd
    rng = np.random.default_rng(B * 1000 + C)
    h, W, b = rng.standard_normal((B, H)), rng.uniform(-1, 1, (C, H)) / np.sqrt(H), rng.uniform(-1, 1, C)
    lab = rng.integers(0, C, B).astype(np.int32)
    if B > 2:
        lab[1] = -1                                   # a row without a target
    h, W, b = (a.astype(np.float32) for a in (h, W, b))
    dev = lambda a: torch.from_numpy(a).cuda()
    loss, dh, dW, db = Bd.xent_head_fwd_bwd(dev(h), dev(W), dev(b), dev(lab))
    h64, W64 = h.astype(np.float64), W.astype(np.float64)
    z = h64 @ W64.T + b.astype(np.float64)
    z -= z.max(axis=1, keepdims=True)
    lse = np.log(np.exp(z).sum(axis=1))
    d = np.exp(z - lse[:, None])
    has = lab >= 0
    want = np.where(has, lse - z[np.arange(B), np.where(has, lab, 0)], 0.0).sum() / B
    d[np.arange(B)[has], lab[has]] -= 1.0
    d /= B
    # fp32 sums of at most 8192 terms; exp through the fast intrinsic: 2 ulp + 1.2e-7 * |argument| (< 10 here)
    assert abs(float(loss) - want) < 2e-5 * max(1.0, abs(want))
    for got, ref in ((dh, d @ W64), (dW, d.T @ h64), (db, d.sum(axis=0))):
        assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref) + 1e-9
