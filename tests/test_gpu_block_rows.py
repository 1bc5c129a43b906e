"""Both layers' row work in one pass (the default block forward) against a pass per layer and against the oracle."""
import pytest
import torch

from oracle import caat_oracle as O
from paper_2506_19645_b200 import caat, synthetic
from tests import gpu_harness as G
from tests.helpers import assert_close, f64

pytestmark = pytest.mark.gpu

CASES = [
    # t, T,    h,    ffn,   S,    norm
    (8, 300, 4096, 11008, 2048, 0),     # units dealt inside tokens, planes of a split GEMM
    (8, 700, 4096, 11008, 2867, 0),     # a chunk that straddles the partition
    (4, 1203, 2048, 5632, 0, 0),        # nothing shared; persistent CTAs walk several tokens
    (4, 1203, 1024, 5632, 1024, 1),     # nothing private, LayerNorm
    (2, 500, 8192, 8192, 4096, 0),      # CTAs of 512 threads
    (4, 333, 768, 3072, 384, 0),        # a warp per token, odd token count
    (4, 2001, 768, 3072, 380, 1),       # the same with LayerNorm, persistent CTAs, a straddling chunk
    (4, 333, 1536, 6144, 200, 0),       # fewer than eight warps
    (2, 130, 264, 528, 131, 1),         # chunks past the row end
    (8, 300, 2048, 5632, 1024, 0),      # both layers' GEMMs in one launch, planes of both
    (8, 129, 2048, 5632, 2048, 0),      # the same with nothing private
]


def _run(ctx, d, T, compact, S, norm, in_place=False):
    t, h = ctx.t, ctx.h
    dev = {k: v.cuda() for k, v in d.items()}
    mk = lambda *s, dt=torch.bfloat16: torch.full(s, 7.0, dtype=dt, device="cuda")
    f32 = torch.float32
    o = {"X1": mk(t, T, h), "rstd1": mk(t, T, dt=f32), "X2": mk(t, T, h), "rstd2": mk(t, T, dt=f32)}
    o["mean1"], o["mean2"] = (mk(t, T, dt=f32), mk(t, T, dt=f32)) if norm else (None, None)
    b1, b2 = (dev["beta1"], dev["beta2"]) if norm else (None, None)
    ws = ctx.alloc_workspace(ctx.block_workspace_bytes(T, False))
    if compact:
        R0s, R0p = dev["R0"][0, :, :S].contiguous(), dev["R0"][:, :, S:].contiguous()
        o.update(Hn1s=R0s if in_place else mk(T, S), Hn1p=R0p if in_place else mk(t, T, h - S), Hn2s=mk(T, S), Hn2p=mk(t, T, h - S))
        ctx.block_forward_compact(T, dev["Y_attn"], dev["W_o"], dev["Y_mlp"], dev["W_down"], R0s, R0p, dev["gamma1"], b1,
                                  dev["gamma2"], b2, o["Hn1s"], o["Hn1p"], o["X1"], o["rstd1"], o["mean1"], o["Hn2s"], o["Hn2p"],
                                  o["X2"], o["rstd2"], o["mean2"], ws)
    else:
        R0 = dev["R0"]
        o.update(Hn1=R0 if in_place else mk(t, T, h), Hn2=mk(t, T, h))
        ctx.block_forward(T, dev["Y_attn"], dev["W_o"], dev["Y_mlp"], dev["W_down"], R0, dev["gamma1"], b1, dev["gamma2"], b2,
                          o["Hn1"], o["X1"], o["rstd1"], o["mean1"], o["Hn2"], o["X2"], o["rstd2"], o["mean2"], ws)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == caat.CAAT_OK
    return {k: v for k, v in o.items() if v is not None}


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("t,T,h,ffn,S,norm", CASES)
def test_block_rows_in_one_pass(t, T, h, ffn, S, norm, compact):
    if compact and S % 8:
        S = S // 8 * 8
    w = synthetic.Workload("blk", t, T, h, ffn, S / h, "bf16", "block", False, T + S)
    d = synthetic.block_inputs(w, S)
    g = torch.Generator().manual_seed(5)
    for k in ("gamma1", "gamma2"):
        d[k] = (1 + 0.1 * torch.randn(h, generator=g)).bfloat16()
        d[k.replace("gamma", "beta")] = (0.1 * torch.randn(h, generator=g)).bfloat16()
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S, norm=norm)
    one = _run(ctx, d, T, compact, S, norm)
    again = _run(ctx, d, T, compact, S, norm, in_place=True)        # the first layer's new stream over its residual
    ctx.set_option(caat.CAAT_OPT_BLOCK_OVERLAP, 0)
    two = _run(ctx, d, T, compact, S, norm)
    beta = (f64(d["beta1"]), f64(d["beta2"])) if norm else (None, None)
    fo = O.block_forward(f64(d["Y_attn"]), f64(d["W_o"]), f64(d["Y_mlp"]), f64(d["W_down"]), f64(d["R0"]), f64(d["gamma1"]),
                         f64(d["gamma2"]), *beta, S=S, alpha=ctx.private_scale, norm=norm)
    for k in one:
        assert torch.equal(one[k], again[k]), f"in place: {k}"
        if k.startswith("Hn"):        # sums and one rounding per element: the same on every row kernel
            assert torch.equal(one[k], two[k]), k
        else:
            assert_close(one[k], f64(two[k]), "bf16", k, scale=0.5)
        if not compact or not k.startswith("Hn"):
            assert_close(one[k], fo[k], "bf16", k)
