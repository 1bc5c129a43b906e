"""What the performance of this package is measured on: the calls of the public binding over the range they are used in.

Every case is one pass of a user's program through the layer, block or MLP entry points: a training step's forward and
backward, a prefill's forward, a decode step.  Sizes are those of ``synthetic.WORKLOADS`` (the configurations of the
benchmark) or generic ones beside them: other token counts, ragged ones among them, other synchronisation factors, the
LayerNorm option, the compact residual stream, fp32.

Kinds: ``layer`` (one MLP-down layer), ``block`` (attention-out then MLP-down), ``compact`` (the block on the stream that
stores its shared channels once), ``mlp`` (column-parallel gate|up with SwiGLU, then the MLP-down layer).
"""
from __future__ import annotations

import math

import torch

from paper_2506_19645_b200 import caat, synthetic

F32 = torch.float32


def _case(name, kind, t, T, h, ffn, p, dtype="bf16", norm="rms", backward=True, graph=False):
    return {"name": name, "kind": kind, "t": t, "T": T, "h": h, "ffn": ffn, "p": p, "dtype": dtype, "norm": norm,
            "backward": backward, "graph": graph}


def listed():
    return [
        # the smallest call: one fp32 layer forward (the benchmark's fp32 configuration); latency and host path
        _case("layer_fp32_small", "layer", 2, 128, 256, 1024, 0.5, dtype="f32", backward=False),
        # an fp32 training step with LayerNorm: what a numerics study or a debugging run of the layer uses
        _case("layer_fp32_train_ln", "layer", 4, 2000, 768, 3072, 0.5, dtype="f32", norm="layer"),
        # one decoded token of a 7B block, called eagerly as an unfused serving loop does
        _case("decode_7b_T1", "block", 8, 1, 4096, 11008, 0.5, backward=False),
        # a decode batch replayed from a CUDA graph, the usual serving set-up
        _case("decode_7b_T8_graph", "block", 8, 8, 4096, 11008, 1.0, backward=False, graph=True),
        # a full decode batch, odd size, graph replay
        _case("decode_7b_T61_graph", "block", 8, 61, 4096, 11008, 0.5, backward=False, graph=True),
        # a short chunk of a chunked prefill (also speculative decoding over a batch): ragged token count
        _case("prefill_7b_T300", "block", 8, 300, 4096, 11008, 0.5, backward=False),
        # a training step of the small model's block at its benchmark size
        _case("train_130m", "block", 4, 16384, 768, 3072, 0.5),
        # a micro-batch of the middle model at a low synchronisation factor, LayerNorm
        _case("train_1p1b_p025_ln", "block", 8, 8192, 2048, 5632, 0.25, norm="layer"),
        # a synchronisation factor that is no multiple of anything (the paper trains at p = 0.7), ragged token count
        _case("train_1p1b_p070_T2999", "block", 8, 2999, 2048, 5632, 0.7),
        # the same block on the compact residual stream
        _case("train_compact_1p1b", "compact", 8, 8192, 2048, 5632, 0.5),
        # a whole tensor-parallel MLP, ragged token count
        _case("train_mlp_1p1b_T6001", "mlp", 8, 6001, 2048, 5632, 0.5),
        # the largest: the headline training step
        _case("train_7b", "block", 8, 16384, 4096, 11008, 0.5),
    ]


#: (t, h, ffn) of the benchmark's models, and generic shapes between and beside them
_SHAPES = [(4, 768, 3072), (8, 2048, 5632), (8, 4096, 11008), (2, 1024, 4096), (4, 1536, 6144), (2, 3072, 8192),
           (8, 5120, 13824)]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _factor(rng):
    """Synchronisation factors: mostly the ones the paper reports, the rest anywhere."""
    return rng.choice([0.0, 0.25, 0.5, 0.75, 1.0]) if rng.random() < 0.6 else round(rng.uniform(0.05, 0.95), 2)


def draw(rng):
    what = rng.choice(["fp32", "decode", "decode", "prefill", "prefill", "train", "train", "train", "compact", "mlp"])
    t, h, ffn = rng.choice(_SHAPES)
    p, norm = _factor(rng), rng.choice(["rms", "rms", "layer"])
    c = {"kind": "block", "t": t, "h": h, "ffn": ffn, "p": p, "dtype": "bf16", "norm": norm, "backward": True,
         "graph": False}
    if what == "fp32":
        # CUDA-core arithmetic: a pass of 25 GFLOP is the upper end of what is run in fp32
        c.update(kind="layer", dtype="f32", backward=rng.random() < 0.5)
        top = 25e9 / ((6 if c["backward"] else 2) * ffn * h)
        c["T"] = max(32, min(_log_int(rng, 64, 2048), int(top)))
    elif what == "decode":
        c.update(T=_log_int(rng, 1, 64), backward=False, graph=rng.random() < 0.5)
    elif what == "prefill":
        c.update(T=_log_int(rng, 65, 8192), backward=False)
    else:
        c.update(kind={"train": "block"}.get(what, what), T=_log_int(rng, 256, 16384))
        if what == "compact":      # the compact stream takes partitions on a multiple of eight channels
            c["p"] = rng.choice([0.25, 0.5, 0.75])
        if what == "mlp":
            c["norm"] = "rms"
    if int(h * p) % 8 and c["dtype"] == "bf16":
        c["T"] = min(c["T"], 4096)     # factors off the grid: sizes of fine-tuning batches
    limit = _cost(listed()[-1])
    while _cost(c) > limit:
        c["T"] = int(c["T"] * 0.8)
    return c


# ---- algorithmic work: every tensor of the method once, 2 m n k per product ----
def _widths(c):
    return (c["ffn"],) if c["kind"] in ("layer", "mlp") else (c["h"], c["ffn"])


def work(case):
    c = case
    t, T, h, e = c["t"], c["T"], c["h"], 4 if c["dtype"] == "f32" else 2
    full = t * T * h
    S = int(h * c["p"])
    stream = T * S + t * T * (h - S) if c["kind"] == "compact" else full
    flops = nbytes = 0.0
    if c["kind"] == "mlp":        # column-parallel half: X, A in, Y inside; backward dX, dA out
        A = 2 * c["ffn"] * h
        flops += 2.0 * T * A * (3 if c["backward"] else 1)
        nbytes += e * (full + A + 2 * T * c["ffn"]) + (e * (2 * T * c["ffn"] + full) + 4 * A if c["backward"] else 0)
    for K in _widths(c):
        flops += 2.0 * T * K * h
        nbytes += e * (T * K + K * h + 2 * stream + full)
        if c["backward"]:
            flops += 4.0 * T * K * h
            nbytes += e * (full + 3 * stream + 2 * T * K + K * h) + 4 * K * h
    return {"bytes": nbytes, "flops": flops}


def _cost(c):
    w = work(c)
    return max(w["bytes"] / 6.4e12, w["flops"] / 1.4e15)


def tolerance(case):
    """About four times what the path differs by from itself in 64 bits (2-norm; largest entry): fp32 5.8e-7 and 6.6e-6
    (sums of hundreds to thousands of products), bf16 3.1e-3 and 1.8e-2 (every partial sum and stored tensor is rounded
    to 8 bits, and the second layer's gradients carry the first one's roundings)."""
    if case["dtype"] == "f32":
        return {"rel": 3e-6, "max": 3e-5}
    return {"rel": 1e-2, "max": 7e-2}


# ---- what a program has in hand before the call ----
def _empty(*shape, dt=torch.bfloat16):
    return torch.empty(*shape, dtype=dt, device="cuda")


def prepare(case, seed):
    c = dict(case)
    t, T, h, p = c["t"], c["T"], c["h"], c["p"]
    ctx = caat.Context(h, c["ffn"], t, p, c["dtype"])
    ln = c["norm"] == "layer"
    if ln:
        ctx.set_option(caat.CAAT_OPT_NORM, caat.LAYERNORM)
    S, td, bwd = ctx.shared_channels, ctx.torch_dtype, c["backward"]
    w = synthetic.Workload("", t, T, h, c["ffn"], p, c["dtype"], c["kind"], bwd, seed)
    ka, km = ctx.k_r(caat.CAAT_ATTN_OUT), ctx.k_r(caat.CAAT_MLP_DOWN)
    mk = lambda *s: _empty(*s, dt=td)  # noqa: E731
    fk = lambda *s: _empty(*s, dt=F32)  # noqa: E731
    st = {"case": c, "ctx": ctx}
    if c["kind"] == "layer":
        i = synthetic.layer_inputs(t, T, h, km, c["dtype"], seed=seed, S=S, backward=bwd, device="cuda")
        o = ctx.alloc_forward_outputs(T)
        if bwd:
            o.update(ctx.alloc_backward_outputs(caat.CAAT_MLP_DOWN, T))
        nbytes = ctx.workspace_bytes(caat.CAAT_MLP_DOWN, T, bwd)
    elif c["kind"] == "mlp":
        i = synthetic.mlp_inputs(w, S, device="cuda")
        o = ctx.alloc_forward_outputs(T)
        o.update({"pre": mk(t, T, 2 * km), "Y": mk(t, T, km)})
        nbytes = ctx.workspace_bytes(caat.CAAT_MLP_DOWN, T, bwd)
        if bwd:
            o.update(ctx.alloc_backward_outputs(caat.CAAT_MLP_DOWN, T))
            o.update({"dX": mk(t, T, h), "dA": fk(t, 2 * km, h)})
            nbytes = max(nbytes, ctx.colpar_workspace_bytes(caat.CAAT_ACT_SWIGLU, 2 * km, T))
    else:
        i = synthetic.block_inputs(w, S, device="cuda")
        o = {"rstd1": fk(t, T), "rstd2": fk(t, T), "X1": mk(t, T, h), "X2": mk(t, T, h)}
        if ln:
            o.update({"mean1": fk(t, T), "mean2": fk(t, T)})
        if c["kind"] == "compact":
            for name in ("R0", "dHn2"):
                if name in i:
                    x = i.pop(name)
                    i[name + "s"], i[name + "p"] = x[0, :, :S].contiguous(), x[:, :, S:].contiguous()
            streams = ["Hn1", "Hn2"] + (["dHn1", "dR0"] if bwd else [])
            o.update({n + "s": mk(T, S) for n in streams})
            o.update({n + "p": mk(t, T, h - S) for n in streams})
        else:
            o.update({n: mk(t, T, h) for n in ["Hn1", "Hn2"] + (["dHn1", "dR0"] if bwd else [])})
        if bwd:
            o.update({"dY_attn": mk(t, T, ka), "dW_o": fk(t, h, ka), "dY_mlp": mk(t, T, km), "dW_down": fk(t, h, km),
                      "dgamma1": fk(h), "dgamma2": fk(h)})
            if ln:
                o.update({"dbeta1": fk(h), "dbeta2": fk(h)})
        nbytes = ctx.block_workspace_bytes(T, bwd)
    # gains near one and, for LayerNorm, small biases, as in a trained network
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1)
    for name in [n for n in i if n.startswith("gamma")]:
        i[name] = (1.0 + 0.1 * torch.randn(h, generator=gen, device="cuda")).to(td)
        if ln:
            i[name.replace("gamma", "beta")] = (0.1 * torch.randn(h, generator=gen, device="cuda")).to(td)
        else:
            i.pop(name.replace("gamma", "beta"), None)
    st["in"], st["out"] = i, {k: v for k, v in o.items() if v is not None}
    st["ws"] = ctx.alloc_workspace(nbytes)
    if c["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _pass(st)
        torch.cuda.current_stream().wait_stream(side)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            _pass(st)
        st["replay"] = g
    return st


# ---- one pass ----
def _layer(st):
    c, i, o, ctx = st["case"], st["in"], st["out"], st["ctx"]
    layer, T = caat.CAAT_MLP_DOWN, c["T"]
    ctx.rowpar_forward(layer, T, i["Y"], i["W"], i["R"], i["gamma"], i.get("beta"), o["Hn"], o["X"], o["rstd"],
                       o.get("mean"), st["ws"])
    if c["backward"]:
        ctx.rowpar_backward(layer, T, i["dX"], i["dHn"], i["Y"], i["W"], o["Hn"], o["rstd"], o.get("mean"), i["gamma"],
                            o["dY"], o["dW"], o["dR"], o["dgamma"], o.get("dbeta"), st["ws"])


def _mlp(st):
    c, i, o, ctx = st["case"], st["in"], st["out"], st["ctx"]
    layer, T, act = caat.CAAT_MLP_DOWN, c["T"], caat.CAAT_ACT_SWIGLU
    n_out = 2 * ctx.k_r(layer)
    ctx.colpar_forward(act, n_out, T, i["X"], i["A"], o["pre"], o["Y"])
    ctx.rowpar_forward(layer, T, o["Y"], i["B"], i["R"], i["gamma"], None, o["Hn"], o["X"], o["rstd"], None, st["ws"])
    if c["backward"]:
        ctx.rowpar_backward(layer, T, i["dXout"], i["dHn"], o["Y"], i["B"], o["Hn"], o["rstd"], None, i["gamma"], o["dY"],
                            o["dW"], o["dR"], o["dgamma"], None, st["ws"])
        ctx.colpar_backward(act, n_out, T, o["dY"], i["X"], i["A"], o["pre"], o["dX"], o["dA"], st["ws"])


def _block(st):
    c, i, o, ctx, ws, T = st["case"], st["in"], st["out"], st["ctx"], st["ws"], st["case"]["T"]
    m1, m2 = o.get("mean1"), o.get("mean2")
    ctx.block_forward(T, i["Y_attn"], i["W_o"], i["Y_mlp"], i["W_down"], i["R0"], i["gamma1"], i.get("beta1"), i["gamma2"],
                      i.get("beta2"), o["Hn1"], o["X1"], o["rstd1"], m1, o["Hn2"], o["X2"], o["rstd2"], m2, ws)
    if c["backward"]:
        ctx.block_backward(T, i["dX1"], i["dX2"], i["dHn2"], i["Y_attn"], i["W_o"], i["Y_mlp"], i["W_down"], o["Hn1"],
                           o["rstd1"], m1, o["Hn2"], o["rstd2"], m2, i["gamma1"], i["gamma2"], o["dY_attn"], o["dW_o"],
                           o["dY_mlp"], o["dW_down"], o["dR0"], o["dHn1"], o["dgamma1"], o.get("dbeta1"), o["dgamma2"],
                           o.get("dbeta2"), ws)


def _compact(st):
    c, i, o, ctx, ws, T = st["case"], st["in"], st["out"], st["ctx"], st["ws"], st["case"]["T"]
    m1, m2 = o.get("mean1"), o.get("mean2")
    ctx.block_forward_compact(T, i["Y_attn"], i["W_o"], i["Y_mlp"], i["W_down"], i["R0s"], i["R0p"], i["gamma1"],
                              i.get("beta1"), i["gamma2"], i.get("beta2"), o["Hn1s"], o["Hn1p"], o["X1"], o["rstd1"], m1,
                              o["Hn2s"], o["Hn2p"], o["X2"], o["rstd2"], m2, ws)
    if c["backward"]:
        ctx.block_backward_compact(T, i["dX1"], i["dX2"], i["dHn2s"], i["dHn2p"], i["Y_attn"], i["W_o"], i["Y_mlp"],
                                   i["W_down"], o["Hn1s"], o["Hn1p"], o["rstd1"], m1, o["Hn2s"], o["Hn2p"], o["rstd2"], m2,
                                   i["gamma1"], i["gamma2"], o["dY_attn"], o["dW_o"], o["dY_mlp"], o["dW_down"], o["dR0s"],
                                   o["dR0p"], o["dHn1s"], o["dHn1p"], o["dgamma1"], o.get("dbeta1"), o["dgamma2"],
                                   o.get("dbeta2"), ws)


def _pass(st):
    {"layer": _layer, "mlp": _mlp, "block": _block, "compact": _compact}[st["case"]["kind"]](st)


def run(state):
    if "replay" in state:
        state["replay"].replay()
    else:
        _pass(state)
    return state["out"]
