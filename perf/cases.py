"""The work that users of this library have it do, as cases that can be timed and compared.

Every case goes through the public entry points (`train_step`, `binding`).  Four kinds:

  train    one training step of a GRU whose layers are solved one after the other: input projection, forward solve, loss
           head, adjoint solve, weight gradients, optimiser update.  `serial` selects the exact sweep + BPTT instead of
           MGRIT; `graph` replays the step from a CUDA graph, as a training loop with fixed shapes does, otherwise every
           step is launched from the host.
  stack    the same up to the gradients, with all layers in one state and one MGRIT cycle for the stack.
  lstm     forward solve, adjoint solve and gradients of one Implicit-LSTM layer.
  forward  the forward solve alone (inference).

Inputs are seeded random sequences: the repository's parameters U(-1/sqrt(H), 1/sqrt(H)) and unit-normal features, ReLU'd
where they stand for the outputs of a convolutional network (dense, half zeros).
"""
from __future__ import annotations

import math

import torch

from paper_2203_04738_b200 import binding as B
from paper_2203_04738_b200 import train_step as TS
from paper_2203_04738_b200.synthetic import Workload

FP32, TF32, BF16 = B.OPERANDS_FP32, B.OPERANDS_TF32, B.OPERANDS_BF16
DEFAULTS = dict(kind="train", layers=1, cf=4, levels=3, fwd=2, adj=2, relax_fine=0, relax_coarse=1, operands=BF16, cell=1,
                classes=51, relu=True, adam=False, serial=False, graph=False)


def _case(name=None, **kw):
    c = dict(DEFAULTS, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest workload of the repository, launched from the host: launches and host work are all there is
        _case("tiny_fp32", T=64, B=2, I=16, H=32, levels=2, operands=FP32, classes=8, relu=False),
        # short clips at fp32 tolerances on the tensor cores (three-term tf32 split), launched from the host
        _case("clip_tf32", T=128, B=16, I=512, H=256, levels=2, relax_fine=1, operands=TF32),
        # wearable-sensor sequences of the paper's first experiment: 9 channels and 100 units rounded up to multiples of 8, batch
        # of 100, two layers, two forward cycles and one backward cycle, Adam, plain fp32
        _case("sensor_fp32", T=128, B=100, I=16, H=104, layers=2, adj=1, operands=FP32, classes=6, relu=False, adam=True),
        # the paper's video experiment: ResNet18-like features, batch of 100 (does not divide a 128-row tile), two layers, Adam
        _case("video_b100", T=128, B=100, I=512, H=1024, layers=2, adj=1, adam=True),
        # mid-sized training step, replayed from a graph
        _case("medium", T=1024, B=32, I=1024, H=512, graph=True),
        # long sequences, small batch: four levels with coarsening by eight
        _case("long", T=4096, B=8, I=2048, H=1024, cf=8, levels=4, fwd=3, adj=3, graph=True),
        # the benchmark's default: two layers of 1024 units over 2048 steps
        _case("train", T=2048, B=32, I=2048, H=1024, layers=2, graph=True),
        # the exact alternative for short sequences: serial sweep + back-propagation through time, one dependent step after another
        _case("serial_bptt", T=512, B=8, I=2048, H=1024, serial=True, graph=True),
        # inference on one stream of ragged length (1000 is no multiple of 16), launched from the host
        _case("infer_b1", kind="forward", T=1000, B=1, I=1024, H=512),
        # odd everything: ragged length, batch that does not divide 128, hidden width of three tiles, FCF on every level
        _case("odd_ragged", T=997, B=24, I=144, H=192, relax_fine=1),
        # two layers in one state and one cycle for the stack
        _case("stack", kind="stack", T=512, B=32, I=1024, H=512, layers=2),
        # one Implicit-LSTM layer of the benchmark's LSTM leg
        _case("lstm", kind="lstm", T=2048, B=32, I=2048, H=1024),
    ]


def draw(rng):
    lg = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    while True:
        kind = rng.choice(["train"] * 6 + ["forward", "forward", "stack", "lstm"])
        operands = rng.choice([BF16, BF16, BF16, TF32, FP32])
        if kind == "stack" and operands == TF32:
            operands = BF16                        # (the stacked calls serve fp32 and bf16 operands)
        cf = rng.choice([2, 4, 4, 4, 8])
        levels = rng.choice([2, 3, 3, 4])
        T, Bn = lg(64, 4096), rng.choice([1, 2, 8, 16, 24, 32, 40, 64, 100, 128, lg(1, 128)])
        if operands == FP32:
            H, I = 8 * lg(4, 32), 8 * lg(2, 64)
        else:
            H, I = 64 * lg(1, 16), 16 * lg(1, 128)
            if T * Bn % 8:
                T = max(8, T // 8 * 8)             # (the tensor-core engines need whole groups of eight rows)
        if T // cf ** (levels - 1) < 2:
            continue
        c = _case(kind=kind, T=T, B=Bn, I=I, H=H, cf=cf, levels=levels, operands=operands, fwd=rng.choice([2, 2, 3]), adj=rng.choice([1, 2, 2]),
                  relax_fine=rng.choice([0, 0, 1]), relax_coarse=rng.choice([0, 1, 1]), relu=rng.random() < 0.7,
                  classes=rng.choice([6, 51, 400]))
        if kind in ("train", "stack"):
            c["layers"] = 2 if kind == "stack" else rng.choice([1, 1, 2])
        if kind == "train":
            c.update(graph=rng.random() < 0.5, serial=rng.random() < 0.15)
            c["adam"] = not c["graph"] and rng.random() < 0.7     # (a graph would bake in Adam's step count)
        # no costlier than the largest listed case; the engines without tensor cores, the exact sweep and the stacked cycle get less
        cap = 4.5e12
        if operands == FP32:
            cap = 6e10
        elif operands == TF32 or kind == "stack":
            cap = 4e11
        if work(c)["flops"] <= cap and not (c["serial"] and T > 2048) and not (kind == "stack" and T > 1024):
            return c


def _flags(c):
    ragged = any(c["T"] % c["cf"] ** l for l in range(c["levels"]))
    return B.FLAG_SKIP_DUPLICATE_FRELAX | (B.FLAG_RAGGED_T if ragged and not c["serial"] else 0)


def _workload(c):
    return Workload("case", T=c["T"], B=c["B"], I=c["I"], H=c["H"], cf=c["cf"], levels=c["levels"], iters_fwd=c["fwd"], iters_adj=c["adj"],
                    relax_fine=c["relax_fine"], relax_coarse=c["relax_coarse"], operands=c["operands"], classes=c["classes"], relu=c["relu"],
                    layers=c["layers"], cell=c["cell"])


def _cfg(c, iters):
    return B.make_cfg(c["T"], c["B"], c["I"], c["H"], cf=c["cf"], levels=c["levels"], iters=iters, cell=c["cell"], relax_fine=c["relax_fine"],
                      relax_coarse=c["relax_coarse"], operands=c["operands"], flags=_flags(c))


def prepare(case, seed):
    """What a training (or serving) program holds before its step: parameters, one batch, buffers and workspaces, the captured
    graph.  (The forward-only case holds its output buffers too; the LSTM and stacked calls allocate theirs on every call.)"""
    c, dev = case, torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    k = 1.0 / math.sqrt(c["H"])
    uni = lambda *s: torch.rand(*s, generator=g, device=dev).mul_(2 * k).sub_(k)
    gates = 4 if c["kind"] == "lstm" else 3
    layers = []
    for l in range(c["layers"]):
        I = c["I"] if l == 0 else c["H"]
        layers.append({"W_ih": uni(gates * c["H"], I), "W_hh": uni(gates * c["H"], c["H"]), "b_ih": uni(gates * c["H"]), "b_hh": uni(gates * c["H"])})
    x = torch.randn(c["T"], c["B"], c["I"], generator=g, device=dev)
    if c["relu"]:
        x.relu_()
    st = {"case": c, "layers": layers, "x": x}
    bytes_ = lambda n: torch.empty(max(n, 1), dtype=torch.uint8, device=dev)
    if c["kind"] == "forward":
        cfg = _cfg(c, c["fwd"])
        cfg.flags |= B.FLAG_GI_CARRIES_COPIES | B.FLAG_GI_F32_UNUSED | B.FLAG_H_LEADS_WITH_H0
        st.update(cfg=cfg, h0=torch.randn(c["B"], c["H"], generator=g, device=dev).mul_(0.3), gi=B.alloc_gi(cfg, dev),
                  h=torch.empty(c["T"] + 1, c["B"], c["H"], device=dev), ws=bytes_(B.workspace_bytes(cfg)[0]))
        return st
    if c["kind"] == "lstm":
        cf_, ca_ = _cfg(c, c["fwd"]), _cfg(c, c["adj"])
        st.update(cfgs=(cf_, ca_), u0=torch.zeros(2, c["B"], c["H"], device=dev), dhT=torch.randn(c["B"], c["H"], generator=g, device=dev),
                  ws_fwd=bytes_(B.lstm_workspace_bytes(cf_)[0]), ws_adj=bytes_(B.lstm_workspace_bytes(ca_)[1]))
        return st
    W_c, b_c = uni(c["classes"], c["H"]), uni(c["classes"])
    labels = torch.randint(0, c["classes"], (c["B"],), generator=g, device=dev, dtype=torch.int32)
    w = _workload(c)
    st.update(w=w, W_c=W_c, b_c=b_c, labels=labels)
    if c["kind"] == "stack":
        cf_, ca_ = _cfg(c, c["fwd"]), _cfg(c, c["adj"])
        st.update(cfgs=(cf_, ca_), h0s=torch.zeros(c["layers"], c["B"], c["H"], device=dev), ws_fwd=bytes_(B.stack_workspace_bytes(cf_, c["layers"])[0]),
                  ws_adj=bytes_(B.stack_workspace_bytes(ca_, c["layers"])[1]), ws_head=bytes_(B.lib.xent_head_workspace_bytes(c["B"], c["classes"])))
        return st
    buf = TS.alloc_buffers(w, c["T"], c["B"], dev, serial=c["serial"], flags=_flags(c))
    adam = TS.AdamState(TS.all_params(layers, W_c, b_c)) if c["adam"] else None
    st.update(h0=torch.zeros(c["B"], c["H"], device=dev), buf=buf, adam=adam)
    if c["graph"]:
        st["step"] = TS.GraphedTrainingStep(w, layers, W_c, b_c, x, st["h0"], labels, buf, adam=adam)
    return st


def run(state):
    st = state
    c = st["case"]
    if c["kind"] == "forward":
        h, _, _ = B.mgrit_gru_forward(st["cfg"], st["layers"][0], st["x"], st["h0"], gi=st["gi"], h=st["h"], ws=st["ws"])
        return {"h": h}
    if c["kind"] == "lstm":
        p = st["layers"][0]
        u, gi, _ = B.mgrit_lstm_forward(st["cfgs"][0], p, st["x"], st["u0"], ws=st["ws_fwd"])
        _, _, o, _ = B.mgrit_lstm_adjoint(st["cfgs"][1], p, st["x"], st["u0"], gi, u, dhT=st["dhT"], want_dx=False, want_du=False, ws=st["ws_adj"])
        return {"u": u, "grads": [o.dW_ih, o.dW_hh, o.db_ih, o.db_hh]}
    if c["kind"] == "stack":
        h, gi0, _ = B.mgrit_gru_stack_forward(st["cfgs"][0], st["layers"], st["x"], st["h0s"], ws=st["ws_fwd"])
        loss, dhT, dWc, dbc = B.xent_head_fwd_bwd(h[-1, -1], st["W_c"], st["b_c"], st["labels"], ws=st["ws_head"])
        _, _, _, outs, _ = B.mgrit_gru_stack_adjoint(st["cfgs"][1], st["layers"], st["x"], st["h0s"], gi0, h, dhT=dhT, want_dx=False, want_dh=False,
                                                     ws=st["ws_adj"])
        return {"loss": loss, "h": h, "grads": [[o.dW_ih, o.dW_hh, o.db_ih, o.db_hh] for o in outs] + [[dWc, dbc]]}
    if c["graph"]:
        loss = st["step"]()
    else:
        loss = TS.training_step(st["w"], st["layers"], st["W_c"], st["b_c"], st["x"], st["h0"], st["labels"], st["buf"], adam=st["adam"])
    return {"loss": loss, "params": TS.all_params(st["layers"], st["W_c"], st["b_c"]), "h": st["buf"].h[-1],
            "grads": [[a.dW_ih, a.dW_hh, a.db_ih, a.db_hh] for a in st["buf"].adj]}


def _points(c, iters, homogeneous):
    """Time points whose cell (or its adjoint) has to be evaluated with a product in `iters` cycles: not the steps that leave
    from the zero initial guess, nor the first F-step of a coarse level (it gives back the v that its right-hand side was made
    of).  homogeneous: the adjoint of a loss on the last state only, zero everywhere before the first coarse solve."""
    if c["serial"]:
        return c["T"]
    n = 0
    for it in range(iters):
        for l in range(c["levels"] - 1):
            N = c["T"] // c["cf"] ** l
            nc = N // c["cf"]
            F = N - nc
            first = (F - nc if it == 0 else 0) if l == 0 else F - nc
            pre = first + (c["relax_fine"] if l == 0 else c["relax_coarse"]) * N + nc + (0 if it == 0 and l == 0 else nc)
            n += F + (0 if homogeneous and it == 0 else pre)
        n += c["T"] // c["cf"] ** (c["levels"] - 1)
    return n


def work(case):
    """Each input read once, each output written once, and the products of the algorithm: projection, cell evaluations of the
    cycles, linearisation on every level, adjoint evaluations, gradient reductions."""
    c = case
    TB, H, B_ = c["T"] * c["B"], c["H"], c["B"]
    g = 4 if c["kind"] == "lstm" else 3
    flops, nbytes = 0.0, 4.0 * TB * c["I"]
    for l in range(c["layers"]):
        I = c["I"] if l == 0 else H
        step = 2.0 * g * H * (H + (I if c["kind"] == "stack" and l > 0 else 0)) * B_
        flops += (0 if c["kind"] == "stack" and l > 0 else 2.0 * TB * g * H * I) + step * _points(c, c["fwd"], False)
        nbytes += 4.0 * g * H * (I + H + 2)
        if c["kind"] == "forward":
            nbytes += 4.0 * TB * H
            continue
        lin = c["T"] if c["serial"] else sum(c["T"] // c["cf"] ** k for k in range(c["levels"]))
        top = l == c["layers"] - 1 or c["kind"] == "stack"
        flops += 2.0 * g * H * H * B_ * lin + step * _points(c, c["adj"], top)
        flops += 2.0 * TB * g * H * (I + H) + (2.0 * TB * g * H * I if l > 0 else 0)
        nbytes += 4.0 * g * H * (I + H + 2) * (2 if c["kind"] == "train" else 1)
    if c["kind"] != "forward":
        nbytes += 4.0 * TB * H * (1 if c["kind"] == "train" else 2)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times what an evaluation at higher precision differs by (2-norm, worst output): bf16 operands against the tf32 split
    2e-3 (states) to 7e-3 (gradients; 1.1e-2 at batch size 1), tf32 split against fp32 4e-6."""
    if case["operands"] == BF16:
        return {"rel": 2e-2}
    return {"rel": 2e-5}
