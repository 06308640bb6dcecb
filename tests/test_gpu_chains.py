"""The bf16 chain kernels at every number of travelling rows (4, 8 and 16, partial and full groups), one and many row groups, widths
with even and uneven splits of the reduction over the warps and units that do not fill the last cluster; the adjoint chains split
by gate and unsplit.  GRU and LSTM serial sweeps and their BPTT against the fp64 oracle, and split against unsplit."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import mgrit_gru_oracle as O
from tests.gpu_util import rel_inf, to_dev

pytestmark = pytest.mark.gpu
SHAPES = [(16, 1, 64), (9, 8, 192), (24, 3, 320), (8, 5, 512), (10, 16, 640), (12, 20, 1024), (8, 33, 256), (16, 9, 128), (6, 4, 1024)]


def _draw(T, B, H, gates):
    rng = np.random.default_rng(T * 1000 + H)
    k = H ** -0.5
    p = {n: rng.uniform(-k, k, s).astype(np.float32) for n, s in dict(W_ih=(gates * H, 16), W_hh=(gates * H, H), b_ih=(gates * H,), b_hh=(gates * H,)).items()}
    return p, rng.standard_normal((T, B, 16)).astype(np.float32), rng.standard_normal((T, 2, B, H)).astype(np.float32)


@pytest.mark.parametrize("c", SHAPES, ids=lambda c: "T{}B{}H{}".format(*c))
@pytest.mark.parametrize("kind", ["gru", "lstm"])
def test_serial_chain_against_the_oracle(c, kind):
    from paper_2203_04738_b200 import binding as Bd
    T, B, H = c
    T += -T % (8 // np.gcd(B, 8))                     # (the engine needs whole groups of eight rows)
    p, x, seed = _draw(T, B, H, 3 if kind == "gru" else 4)
    dev = {n: to_dev(v) for n, v in p.items()}
    P = [p[n].astype(np.float64) for n in ("W_ih", "W_hh", "b_ih", "b_hh")]
    cfg = Bd.make_cfg(T, B, 16, H, cf=2, levels=1, operands=2)
    n0 = Bd.kernel_launches()
    if kind == "gru":
        h0 = np.random.default_rng(5).standard_normal((B, H)).astype(np.float32) * np.float32(0.3)
        h, gi = Bd.gru_serial_forward(cfg, dev, to_dev(x), to_dev(h0))
        n1 = Bd.kernel_launches()
        assert rel_inf(h.cpu().numpy(), O.serial_forward(*P, x.astype(np.float64), h0.astype(np.float64))) < 2e-2
        hn = h.cpu().numpy().astype(np.float64)
        r = Bd.gru_serial_backward(cfg, dev, to_dev(x), to_dev(h0), gi, h, dh_seed=to_dev(seed[:, 0]))
        lam, lam0, g = O.serial_backward(*P, x.astype(np.float64), h0.astype(np.float64), hn, seed[:, 0].astype(np.float64))
        assert rel_inf(r.dh.cpu().numpy(), lam) < 2e-2 and rel_inf(r.dh0.cpu().numpy(), lam0) < 2e-2
        assert rel_inf(r.dW_hh.cpu().numpy(), g["dW_hh"]) < 2e-2
    else:
        u0 = np.random.default_rng(5).standard_normal((2, B, H)).astype(np.float32) * np.float32(0.3)
        u, gi, _ = Bd.mgrit_lstm_forward(cfg, dev, to_dev(x), to_dev(u0))
        n1 = Bd.kernel_launches()
        uref = O.lstm_serial_forward(*P, x.astype(np.float64), u0.astype(np.float64))
        assert rel_inf(u.cpu().numpy(), uref) < 2e-2
        un = u.cpu().numpy().astype(np.float64)
        du, du0, o, _ = Bd.mgrit_lstm_adjoint(cfg, dev, to_dev(x), to_dev(u0), gi, u, du_seed=to_dev(seed))
        ref = O.lstm_serial_backward(*P, x.astype(np.float64), u0.astype(np.float64), un, seed.astype(np.float64))
        assert rel_inf(du.cpu().numpy(), ref[0]) < 2e-2
        assert rel_inf(o.dW_hh.cpu().numpy(), ref[2]["dW_hh"]) < 2e-2
    assert n1 - n0 < 10                                # one chain, not one launch per step
    assert Bd.last_device_status() == 0


CHILD = r"""
import sys, numpy as np, torch
from paper_2203_04738_b200 import binding as B
from tests.test_gpu_chains import SHAPES, _draw
from tests.gpu_util import to_dev
out = {}
for i, (T, Bz, H) in enumerate([(24, 9, 640), (16, 20, 1024), (16, 4, 576)]):
    for gates in (3, 4):
        p, x, seed = _draw(T, Bz, H, gates)
        dev = {n: to_dev(v) for n, v in p.items()}
        cfg = B.make_cfg(T, Bz, 16, H, cf=2, levels=1, operands=2)
        if gates == 3:
            h0 = torch.zeros(Bz, H, device="cuda")
            h, gi = B.gru_serial_forward(cfg, dev, to_dev(x), h0)
            out[f"g{i}"] = B.gru_serial_backward(cfg, dev, to_dev(x), h0, gi, h, dh_seed=to_dev(seed[:, 0])).dh.cpu().numpy()
        else:
            u0 = torch.zeros(2, Bz, H, device="cuda")
            u, gi, _ = B.mgrit_lstm_forward(cfg, dev, to_dev(x), u0)
            out[f"l{i}"] = B.mgrit_lstm_adjoint(cfg, dev, to_dev(x), u0, gi, u, du_seed=to_dev(seed))[0].cpu().numpy()
assert B.last_device_status() == 0
np.savez(sys.argv[1], **out)
"""


def test_split_by_gate_agrees_with_unsplit(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    outs = []
    for flag in ("1", "0"):
        out = str(tmp_path / f"c{flag}.npz")
        env = dict(os.environ, MGRIT_GRU_CHAIN_SPLIT=flag, PYTHONPATH=root)
        subprocess.run([sys.executable, "-c", CHILD, out], check=True, env=env, cwd=root, timeout=600)
        outs.append(np.load(out))
    a, b = outs
    for k in a.files:
        # the same products summed in another order; a few operands round to the other side of a bf16 tie (2^-9)
        assert np.linalg.norm(a[k] - b[k]) <= 2e-3 * np.linalg.norm(b[k]), k
