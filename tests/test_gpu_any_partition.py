"""Partitions off the 8-channel grid on the tensor-core and few-token paths.

The tensor-core GEMMs start the private channels at S rounded down to 8: extra scratch columns in the forward, zero-filled
weight rows in the data gradient, rows left out of the store in the weight gradient.  The few-token row kernels sum the
chunk that straddles the partition both ways.  Checked against the fp64 oracle at the partition's extremes."""
import pytest
import torch

from oracle import caat_oracle as O
from paper_2506_19645_b200 import caat, synthetic
from tests import gpu_harness as G
from tests.helpers import assert_close, f64
from tests.test_gpu_parity import _check_backward, _check_forward, _layer_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,T,h,ffn,layer,S,alpha,norm", [
    (8, 300, 2048, 5632, caat.CAAT_MLP_DOWN, 1433, None, 0),    # p = 0.7: pair tiles
    (8, 130, 4096, 11008, caat.CAAT_MLP_DOWN, 2867, None, 1),
    (4, 257, 768, 3072, caat.CAAT_ATTN_OUT, 1, None, 0),        # one shared channel: the private part starts at column 0
    (4, 257, 768, 3072, caat.CAAT_ATTN_OUT, 767, 1.0, 0),       # one private channel, no scaled weights
    (4, 100, 768, 3072, caat.CAAT_MLP_DOWN, 257, None, 0),      # just past a tile edge
    (2, 3000, 256, 1024, caat.CAAT_ATTN_OUT, 131, None, 0),     # small weight gradient: split-K partials
    (2, 70, 16, 64, caat.CAAT_ATTN_OUT, 11, None, 0),           # K_r = 8, a single tile
    (8, 1, 4096, 11008, caat.CAAT_MLP_DOWN, 2867, None, 0),     # few tokens, one cluster per token
    (4, 5, 768, 3072, caat.CAAT_ATTN_OUT, 3, None, 1),
    (8, 64, 1024, 4096, caat.CAAT_MLP_DOWN, 1017, None, 0),     # many rows: CTA per row / two CTAs per SM
    (3, 33, 264, 792, caat.CAAT_ATTN_OUT, 259, 0.5, 1),         # fewer than 8 private channels
    (8, 300, 2048, 5632, caat.CAAT_MLP_DOWN, 1433, 0.0, 0),     # private scale 0: no gradient reaches the private rows
    (8, 300, 2048, 5632, caat.CAAT_MLP_DOWN, 1432, 0.0, 0),     # the same on the grid
    (2, 3000, 256, 1024, caat.CAAT_ATTN_OUT, 131, 0.0, 1),      # the same through split-K partials
    (4, 257, 768, 3072, caat.CAAT_ATTN_OUT, 381, -1.5, 0),      # a negative scale, on the epilogues
    (4, 257, 768, 3072, caat.CAAT_ATTN_OUT, 384, -4096.0, 0),   # the same on the scaled weights
])
def test_layer_with_a_partition_off_the_grid(t, T, h, ffn, layer, S, alpha, norm):
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S, alpha=alpha, norm=norm)
    d = _layer_case(t, T, h, ctx.k_r(layer), "bf16", S, seed=T + S, backward=True)
    g = torch.Generator().manual_seed(5)
    d["gamma"] = (1 + 0.1 * torch.randn(h, generator=g)).bfloat16()
    d["beta"] = (0.1 * torch.randn(h, generator=g)).bfloat16()
    _check_forward(ctx, layer, d, "bf16")
    _check_backward(ctx, layer, d, "bf16")


@pytest.mark.parametrize("T,S", [(1, 1433), (13, 1433), (64, 2041), (64, 5)])
def test_two_layer_few_token_block_with_a_partition_off_the_grid(T, S):
    t, h, ffn = 8, 2048, 5632
    w = synthetic.Workload("blk", t, T, h, ffn, S / h, "bf16", "block", False, T + S)
    d = synthetic.block_inputs(w, S)
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S)
    dev = {k: v.cuda() for k, v in d.items()}
    mk = lambda *s, dt=torch.bfloat16: torch.empty(*s, dtype=dt, device="cuda")
    Hn1, X1, Hn2, X2 = (mk(t, T, h) for _ in range(4))
    rstd1, rstd2 = mk(t, T, dt=torch.float32), mk(t, T, dt=torch.float32)
    ws = ctx.alloc_workspace(ctx.block_workspace_bytes(T, False))
    ctx.block_forward(T, dev["Y_attn"], dev["W_o"], dev["Y_mlp"], dev["W_down"], dev["R0"], dev["gamma1"], None,
                      dev["gamma2"], None, Hn1, X1, rstd1, None, Hn2, X2, rstd2, None, ws)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == caat.CAAT_OK
    fo = O.block_forward(f64(d["Y_attn"]), f64(d["W_o"]), f64(d["Y_mlp"]), f64(d["W_down"]), f64(d["R0"]),
                         f64(d["gamma1"]), f64(d["gamma2"]), S=S, alpha=ctx.private_scale)
    for name, g in (("Hn1", Hn1), ("X1", X1), ("Hn2", Hn2), ("X2", X2), ("rstd1", rstd1), ("rstd2", rstd2)):
        assert_close(g, fo[name], "bf16", name)


@pytest.mark.parametrize("T", [1, 64])
def test_few_tokens_on_a_workspace_made_for_more(T):
    # 100 tokens need less scratch than the fp32 planes of a few; such a call goes without them
    t, h, ffn, S = 8, 2048, 5632, 1433
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S)
    w = synthetic.Workload("blk", t, T, h, ffn, S / h, "bf16", "block", False, T)
    d = synthetic.block_inputs(w, S)
    dev = {k: v.cuda() for k, v in d.items()}
    mk = lambda *s, dt=torch.bfloat16: torch.empty(*s, dtype=dt, device="cuda")
    Hn1, X1, Hn2, X2 = (mk(t, T, h) for _ in range(4))
    rstd1, rstd2 = mk(t, T, dt=torch.float32), mk(t, T, dt=torch.float32)
    small = ctx.alloc_workspace(ctx.workspace_bytes(caat.CAAT_MLP_DOWN, 100, False))
    assert T == 1 or small.numel() < ctx.workspace_bytes(caat.CAAT_MLP_DOWN, T, False)
    fo = O.block_forward(f64(d["Y_attn"]), f64(d["W_o"]), f64(d["Y_mlp"]), f64(d["W_down"]), f64(d["R0"]),
                         f64(d["gamma1"]), f64(d["gamma2"]), S=S, alpha=ctx.private_scale)
    ctx.block_forward(T, dev["Y_attn"], dev["W_o"], dev["Y_mlp"], dev["W_down"], dev["R0"], dev["gamma1"], None,
                      dev["gamma2"], None, Hn1, X1, rstd1, None, Hn2, X2, rstd2, None, small)
    torch.cuda.synchronize()
    for name, g in (("Hn1", Hn1), ("X1", X1), ("Hn2", Hn2), ("X2", X2)):
        assert_close(g, fo[name], "bf16", name)
    ctx.rowpar_forward(caat.CAAT_ATTN_OUT, T, dev["Y_attn"], dev["W_o"], dev["R0"], dev["gamma1"], None, Hn2, X2, rstd2, None, small)
    torch.cuda.synchronize()
    assert_close(Hn2, fo["Hn1"], "bf16", "Hn1 of the layer call")
    assert ctx.last_device_status() == caat.CAAT_OK
