"""The default block backward - both layers' row work in one pass, their four gradient products in one launch, or both -
against the layers one after the other and against the oracle."""
import pytest
import torch

from oracle import caat_oracle as O
from paper_2506_19645_b200 import caat, synthetic
from tests import gpu_harness as G
from tests.helpers import assert_close, f64

pytestmark = pytest.mark.gpu

CASES = [
    # t, T,   h,    ffn,  S,    norm, stream gradient given
    (8, 300, 2048, 5632, 1024, 0, True),     # two chunks per thread, 128 threads
    (4, 621, 2048, 5632, 1433, 0, True),     # a chunk that straddles the partition, several tokens per CTA
    (2, 170, 4096, 8192, 2048, 0, True),     # two chunks per thread, 256 threads
    (2, 170, 3072, 6144, 1000, 1, True),     # 384 threads, LayerNorm
    (2, 333, 1536, 3072, 1536, 0, True),     # nothing private, 192 threads
    (4, 701, 1024, 4096, 0, 1, False),       # nothing shared, no stream gradient
    (4, 130, 768, 3072, 380, 0, False),      # three warps per token
    (2, 2050, 512, 1024, 256, 0, True),      # two tokens per CTA, many rounds
    (2, 77, 272, 544, 128, 1, True),         # chunks past the row end
    # rows of the layers one after the other, their four gradient products in one launch
    (8, 300, 2048, 5632, 1024, 1, True),
    (2, 257, 2048, 5632, 2048, 1, False),    # nothing private
    (2, 129, 5120, 10240, 0, 0, True),       # nothing shared
    (4, 200, 2048, 4096, 1003, 1, True),     # a partition off the 8-channel grid
]


def _run(ctx, d, sv, T, compact, S, norm, dh, in_place=()):
    """in_place: "dHn1" puts the second layer's residual gradient over the stream gradient, "dR0" the first one's over that."""
    t, h = ctx.t, ctx.h
    dev = {k: v.cuda() for k, v in d.items()}
    f32 = torch.float32
    mk = lambda *s, dt=torch.bfloat16: torch.full(s, 7.0, dtype=dt, device="cuda")
    ka, km = ctx.k_r(caat.CAAT_ATTN_OUT), ctx.k_r(caat.CAAT_MLP_DOWN)
    o = {"dY_attn": mk(t, T, ka), "dW_o": mk(t, h, ka, dt=f32), "dY_mlp": mk(t, T, km), "dW_down": mk(t, h, km, dt=f32),
         "dgamma1": mk(h, dt=f32), "dgamma2": mk(h, dt=f32)}
    o["dbeta1"], o["dbeta2"] = (mk(h, dt=f32), mk(h, dt=f32)) if norm else (None, None)
    r1, m1, r2, m2 = (sv[k].cuda() if sv[k] is not None else None for k in ("rstd1", "mean1", "rstd2", "mean2"))
    ws = ctx.alloc_workspace(ctx.block_workspace_bytes(T, True))
    part = lambda x: (x[0, :, :S].contiguous().cuda(), x[:, :, S:].contiguous().cuda())
    if compact:
        o.update(dR0s=mk(T, S), dR0p=mk(t, T, h - S), dHn1s=mk(T, S), dHn1p=mk(t, T, h - S))
        dHs, dHp = part(d["dHn2"]) if dh else (None, None)
        if "dHn1" in in_place:
            o["dHn1s"], o["dHn1p"] = dHs, dHp
        if "dR0" in in_place:
            o["dR0s"], o["dR0p"] = o["dHn1s"], o["dHn1p"]
        ctx.block_backward_compact(T, dev["dX1"], dev["dX2"], dHs, dHp, dev["Y_attn"], dev["W_o"], dev["Y_mlp"], dev["W_down"],
                                   *part(sv["Hn1"]), r1, m1, *part(sv["Hn2"]), r2, m2, dev["gamma1"], dev["gamma2"], o["dY_attn"],
                                   o["dW_o"], o["dY_mlp"], o["dW_down"], o["dR0s"], o["dR0p"], o["dHn1s"], o["dHn1p"], o["dgamma1"],
                                   o["dbeta1"], o["dgamma2"], o["dbeta2"], ws)
    else:
        o.update(dR0=mk(t, T, h), dHn1=mk(t, T, h))
        if "dHn1" in in_place:
            o["dHn1"] = dev["dHn2"]
        if "dR0" in in_place:
            o["dR0"] = o["dHn1"]
        ctx.block_backward(T, dev["dX1"], dev["dX2"], dev["dHn2"] if dh else None, dev["Y_attn"], dev["W_o"], dev["Y_mlp"],
                           dev["W_down"], sv["Hn1"].cuda(), r1, m1, sv["Hn2"].cuda(), r2, m2, dev["gamma1"], dev["gamma2"],
                           o["dY_attn"], o["dW_o"], o["dY_mlp"], o["dW_down"], o["dR0"], o["dHn1"], o["dgamma1"], o["dbeta1"],
                           o["dgamma2"], o["dbeta2"], ws)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == caat.CAAT_OK
    return {k: v for k, v in o.items() if v is not None}


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("t,T,h,ffn,S,norm,dh", CASES)
def test_block_backward_rows_in_one_pass(t, T, h, ffn, S, norm, dh, compact):
    _check(t, T, h, ffn, S, norm, dh, compact)


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("S", [1024, 1003])
@pytest.mark.parametrize("alpha", [0.0, -1.5])
def test_block_backward_at_any_private_scale(alpha, S, compact):
    _check(8, 300, 2048, 5632, S, 0, True, compact, alpha)      # the four gradient products in one launch


def _inputs(t, T, h, ffn, S, norm, compact):
    w = synthetic.Workload("blk", t, T, h, ffn, S / h, "bf16", "block", True, T + S)
    d = synthetic.block_inputs(w, S)
    g = torch.Generator().manual_seed(5)
    for k in ("gamma1", "gamma2"):
        d[k] = (1 + 0.1 * torch.randn(h, generator=g)).bfloat16()
    sv = {}
    for l in ("1", "2"):
        x = torch.randn(t, T, h, generator=g)
        if compact:
            x[:, :, :S] = x[:1, :, :S]
        sv["Hn" + l] = x.bfloat16()
        x = f64(sv["Hn" + l])
        mean = x.mean(2) if norm else 0 * x.mean(2)
        sv["mean" + l] = torch.from_numpy(mean).float() if norm else None
        sv["rstd" + l] = torch.from_numpy(((x - mean[:, :, None]) ** 2).mean(2) ** -0.5).float()
    return d, sv


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("t,T,h,ffn,S,norm", [(8, 300, 2048, 5632, 1024, 0), (2, 2050, 512, 1024, 256, 0), (2, 333, 1536, 3072, 1536, 1),
                                              (4, 701, 1024, 4096, 0, 0)])
def test_block_backward_in_place(t, T, h, ffn, S, norm, compact):
    d, sv = _inputs(t, T, h, ffn, S, norm, compact)
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S, norm=norm)
    run = lambda *where: _run(ctx, d, sv, T, compact, S, norm, True, where)
    want, got = run(), run("dHn1")                # every element of the stream gradient is read before its place is written
    for k in want:
        assert torch.equal(want[k], got[k]), k
    chained = run("dR0"), run("dHn1", "dR0")      # these take the layers one after the other
    ctx.set_option(caat.CAAT_OPT_BLOCK_OVERLAP, 0)
    want = run()
    for got in chained:
        for k in want:
            if not k.startswith("dHn1"):          # overwritten by dR0
                assert torch.equal(want[k], got[k]), k


def _check(t, T, h, ffn, S, norm, dh, compact, alpha=None):
    if compact:
        S = S // 8 * 8
    d, sv = _inputs(t, T, h, ffn, S, norm, compact)
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S, norm=norm, alpha=alpha)
    before = caat.kernel_launches()
    one = _run(ctx, d, sv, T, compact, S, norm, dh)
    mid = caat.kernel_launches()
    ctx.set_option(caat.CAAT_OPT_BLOCK_OVERLAP, 0)
    two = _run(ctx, d, sv, T, compact, S, norm, dh)
    if not (compact and h <= 768 and T > 2000):                   # those keep a pass per layer
        assert caat.kernel_launches() - mid >= mid - before + 2   # one row kernel and one norm-gradient sum less
    z = lambda x: None if x is None else f64(x)
    args = [z(d["Y_attn"]), z(d["W_o"]), z(d["Y_mlp"]), z(d["W_down"])]
    if compact:
        p = lambda x: (f64(x[0, :, :S]), f64(x[:, :, S:]))
        ob = O.block_backward_compact(z(d["dX1"]), z(d["dX2"]), *(p(d["dHn2"]) if dh else (None, None)), *args, *p(sv["Hn1"]),
                                      z(sv["rstd1"]), z(sv["mean1"]), *p(sv["Hn2"]), z(sv["rstd2"]), z(sv["mean2"]), z(d["gamma1"]),
                                      z(d["gamma2"]), S=S, alpha=ctx.private_scale, norm=norm)
    else:
        ob = O.block_backward(z(d["dX1"]), z(d["dX2"]), z(d["dHn2"]) if dh else None, *args, z(sv["Hn1"]), z(sv["rstd1"]),
                              z(sv["mean1"]), z(sv["Hn2"]), z(sv["rstd2"]), z(sv["mean2"]), z(d["gamma1"]), z(d["gamma2"]), S=S,
                              alpha=ctx.private_scale, norm=norm)
    for k in one:
        assert_close(one[k], ob[k], "bf16", k)
        assert_close(one[k], f64(two[k]), "bf16", k, scale=0.5)   # another order of the same fp32 sums, each rounded to bf16
