"""fp32 products on the bf16 tensor cores (operands split in three parts): tiles, pairs and clusters at their edges, both
operand majors, 16-byte and element-wise loads, accuracy against 64 bits beside the CUDA-core path, values that are not finite."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2506_19645_b200 import caat, synthetic
from tests import gpu_harness as G
from tests.test_gpu_parity import _check_backward, _check_forward, _layer_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,T,h,ffn,layer,S", [
    (4, 64, 768, 3072, caat.CAAT_MLP_DOWN, 384),      # few tokens: the weights on the 128-row side, contractions over clusters
    (4, 257, 768, 3072, caat.CAAT_MLP_DOWN, 384),     # one row past a pair's tile
    (4, 999, 768, 3000, caat.CAAT_MLP_DOWN, 285),     # K_r = 750 and an odd partition: element-wise loads, remainders everywhere
    (4, 640, 768, 3088, caat.CAAT_MLP_DOWN, 380),     # K_r = 772: 16-byte loads with remainders
    (2, 777, 1032, 4104, caat.CAAT_MLP_DOWN, 1032),   # nothing private
    (2, 777, 1032, 4104, caat.CAAT_MLP_DOWN, 0),      # nothing shared
    (1, 1500, 1032, 2064, caat.CAAT_MLP_DOWN, 8),     # one rank, a shared tile of 8 columns
    (8, 300, 2048, 5632, caat.CAAT_MLP_DOWN, 1024),   # more tiles than clusters: partial tiles and the next item's operands
    (2, 3000, 1024, 4096, caat.CAAT_ATTN_OUT, 512),   # tiles for several rounds
])
def test_f32_layer(t, T, h, ffn, layer, S):
    ctx = G.make_ctx(t, h, ffn, "f32", S=S)
    d = _layer_case(t, T, h, ctx.k_r(layer), "f32", S, seed=T + S, backward=True)
    caat.profile_begin(64)
    _check_forward(ctx, layer, d, "f32")
    _check_backward(ctx, layer, d, "f32")
    assert "gemm_cuda_core" not in caat.profile_end()


@pytest.mark.parametrize("t,T,h,ffn,S,stays", [
    (1, 64, 128, 16384, 64, "forward"),         # two row tiles and a contraction of 256 chunks
    (1, 100, 256, 8192, 256, "forward"),
    (1, 1024, 128, 16384, 64, ""),              # the same contraction, tiles for all SMs
    (8, 64, 1024, 2816, 921, ""),               # short contractions, element by element: the results' contiguous axis on the lanes
])
def test_products_that_stay_on_the_cuda_cores(t, T, h, ffn, S, stays):
    """Of the layer's three products the named one and no other; every output against the CUDA cores alone."""
    layer, out, kinds = caat.CAAT_MLP_DOWN, [], None
    for force in (True, False):
        ctx = G.make_ctx(t, h, ffn, "f32", S=S, force_simt=force)
        d = synthetic.layer_inputs(t, T, h, ctx.k_r(layer), "f32", seed=T, S=S, backward=True, device="cuda")
        o = ctx.alloc_forward_outputs(T)
        o.update(ctx.alloc_backward_outputs(layer, T))
        ws = ctx.alloc_workspace(ctx.workspace_bytes(layer, T, True))
        caat.profile_begin(64)
        ctx.rowpar_forward(layer, T, d["Y"], d["W"], d["R"], d["gamma"], None, o["Hn"], o["X"], o["rstd"], None, ws)
        ctx.rowpar_backward(layer, T, d["dX"], d["dHn"], d["Y"], d["W"], o["Hn"], o["rstd"], None, d["gamma"], o["dY"], o["dW"],
                            o["dR"], o["dgamma"], None, ws)
        torch.cuda.synchronize()
        assert ctx.last_device_status() == caat.CAAT_OK
        kinds = {k for k in caat.profile_end() if "gemm" in k}
        out.append(o)
    here = {"tc_gemm_forward", "tc_gemm_dgrad", "tc_gemm_wgrad"} - {"tc_gemm_" + stays}
    assert kinds == here | ({"gemm_cuda_core"} if stays else set())
    for name in ("Hn", "dY", "dW", "dR"):
        a, b = out[0][name].double(), out[1][name].double()
        # chains of up to 16384 products on the CUDA cores: 2^-24 sqrt(16384) / 2 = 3.8e-6 at most, through the norm into the gradients
        assert float((a - b).norm() / a.norm()) < 8e-6, name


def _rel(a, b):
    return float(((a.double().numpy() - b) ** 2).sum() ** 0.5 / (b ** 2).sum() ** 0.5)


@pytest.mark.parametrize("t,T,h,ffn,p", [(4, 2000, 768, 3072, 0.5), (8, 64, 2048, 5632, 0.91), (2, 300, 1024, 4096, 0.0)])
def test_no_further_from_64_bits_than_fma_chains(t, T, h, ffn, p):
    """The three parts hold all 24 bits and a partial sum of 64 products is added in fp32 registers: 1.0e-7 to 1.4e-7 here, where
    the CUDA-core kernels' chains of FMAs give 1.0e-7 to 5.7e-7."""
    layer, out = caat.CAAT_MLP_DOWN, []
    for force in (True, False):
        ctx = G.make_ctx(t, h, ffn, "f32", p=p, force_simt=force)
        d = _layer_case(t, T, h, ctx.k_r(layer), "f32", ctx.shared_channels, seed=5, backward=True)
        fo = G.oracle_forward(ctx, d)
        Hn, rstd, mean = G.saved_from_oracle(ctx, fo)
        got, gb, ob = G.gpu_forward(ctx, layer, d), G.gpu_backward(ctx, layer, d, Hn, rstd, mean), G.oracle_backward(ctx, d, Hn, rstd, mean)
        out.append([_rel(got["Hn"], fo["Hn"]), _rel(gb["dY"], ob["dY"]), _rel(gb["dW"], ob["dW"])])
    for simt, tensor in zip(*out):
        assert tensor < 2.5e-7 and tensor < 1.1 * simt


@pytest.mark.parametrize("spread", [0, 2])
def test_operands_that_lose_the_most(spread):
    """The square of 1.0038986 (parts 1, 2^-8, -2^-17) loses 2^-24 in the products that are left out, the most any product can.  A
    sum of such products of one sign loses as much, and the accumulator's truncation and the fp32 additions of the partial
    sums come on top: each stays below 2^-24 here (6e-8 and less, measured)."""
    t, T, h, ffn, layer = 1, 2000, 1024, 4096, caat.CAAT_MLP_DOWN
    ctx = G.make_ctx(t, h, ffn, "f32", S=0, alpha=1.0)
    d = _layer_case(t, T, h, ctx.k_r(layer), "f32", 0, seed=1)
    g = torch.Generator().manual_seed(1)
    for n in ("Y", "W"):
        d[n] = torch.ldexp(torch.full_like(d[n], 1.0038986206), torch.randint(-spread, spread + 1, d[n].shape, generator=g))
    d["R"].zero_()
    assert _rel(G.gpu_forward(ctx, layer, d)["Hn"], G.oracle_forward(ctx, d)["Hn"]) < 3 * 2.0 ** -24


def _block_and_column_calls(ctx, T, compact, seed):
    """A block's forward and backward on the layers' scratch, and a column-parallel layer's: every output by name."""
    t, h, S, f32 = ctx.t, ctx.h, ctx.shared_channels, torch.float32
    ka, km = ctx.k_r(caat.CAAT_ATTN_OUT), ctx.k_r(caat.CAAT_MLP_DOWN)
    i = synthetic.block_inputs(synthetic.Workload("", t, T, h, km * t, S / h, "f32", "block", True, seed), S, device="cuda")
    mk = lambda *s: torch.empty(*s, dtype=f32, device="cuda")  # noqa: E731
    part = (lambda x: [x[0, :, :S].contiguous(), x[:, :, S:].contiguous()]) if compact else (lambda x: [x])
    new = (lambda: [mk(T, S), mk(t, T, h - S)]) if compact else (lambda: [mk(t, T, h)])
    ws = ctx.alloc_workspace(ctx.block_workspace_bytes(T, True))
    Hn1, X1, r1, Hn2, X2, r2 = new(), mk(t, T, h), mk(t, T), new(), mk(t, T, h), mk(t, T)
    (ctx.block_forward_compact if compact else ctx.block_forward)(
        T, i["Y_attn"], i["W_o"], i["Y_mlp"], i["W_down"], *part(i["R0"]), i["gamma1"], None, i["gamma2"], None, *Hn1, X1, r1, None,
        *Hn2, X2, r2, None, ws)
    dYa, dWo, dYm, dWd, dR0, dHn1, dg1, dg2 = mk(t, T, ka), mk(t, h, ka), mk(t, T, km), mk(t, h, km), new(), new(), mk(h), mk(h)
    (ctx.block_backward_compact if compact else ctx.block_backward)(
        T, i["dX1"], i["dX2"], *part(i["dHn2"]), i["Y_attn"], i["W_o"], i["Y_mlp"], i["W_down"], *Hn1, r1, None, *Hn2, r2, None,
        i["gamma1"], i["gamma2"], dYa, dWo, dYm, dWd, *dR0, *dHn1, dg1, None, dg2, None, ws)
    n_out, act = 2 * km, caat.CAAT_ACT_SWIGLU
    A = torch.cat([i["W_down"], -i["W_down"]], 2).transpose(1, 2).contiguous()
    pre, Y, dX, dA = mk(t, T, n_out), mk(t, T, km), mk(t, T, h), mk(t, n_out, h)
    ctx.colpar_forward(act, n_out, T, i["R0"], A, pre, Y)
    ctx.colpar_backward(act, n_out, T, i["Y_mlp"], i["R0"], A, pre, dX, dA, ctx.alloc_workspace(ctx.colpar_workspace_bytes(act, n_out, T)))
    torch.cuda.synchronize()
    assert ctx.last_device_status() == caat.CAAT_OK
    return dict(Hn1=Hn1[-1], X1=X1, Hn2=Hn2[-1], X2=X2, Hn1s=Hn1[0], Hn2s=Hn2[0], dYa=dYa, dWo=dWo, dYm=dYm, dWd=dWd, dR0=dR0[-1],
                dR0s=dR0[0], dg1=dg1, dg2=dg2, pre=pre, Y=Y, dX=dX, dA=dA)


@pytest.mark.parametrize("t,T,h,ffn,p,compact", [(4, 700, 768, 3072, 0.5, False), (4, 700, 768, 3072, 0.5, True), (2, 333, 1032, 4128, 0.3, False)])
def test_blocks_and_column_parallel_layers(t, T, h, ffn, p, compact):
    """The other entry points' products go the same way, none to the CUDA cores, and give what those give to both sides' rounding."""
    out = []
    for force in (True, False):
        ctx = G.make_ctx(t, h, ffn, "f32", p=p, force_simt=force)
        caat.profile_begin(64)
        out.append(_block_and_column_calls(ctx, T, compact, seed=T))
        kinds = set(caat.profile_end())
        gemms = {k for k in kinds if "gemm" in k}
        assert gemms == ({"gemm_cuda_core"} if force else {"tc_gemm_forward", "tc_gemm_dgrad", "tc_gemm_wgrad"})
    for name, want in out[0].items():
        got = out[1][name]
        # chains of up to 4128 products: 6e-7 each side at most, twice through the block's second layer
        assert float((got - want).double().norm() / want.double().norm()) < 3e-6, name


@pytest.mark.parametrize("ey,ew", [(-120, 100), (100, -120), (-126, 0), (0, -126), (-100, -30), (-70, -70), (60, 45)])
def test_small_and_large_operands(ey, ew):
    """Operands near the smallest normal numbers keep all their bits, products that are not normal and sums that are large
    come out as the CUDA cores' chains give them."""
    t, T, h, ffn, layer, out = 4, 300, 768, 3072, caat.CAAT_MLP_DOWN, []
    for force in (True, False):
        ctx = G.make_ctx(t, h, ffn, "f32", p=0.5, force_simt=force)
        d = _layer_case(t, T, h, ctx.k_r(layer), "f32", ctx.shared_channels, seed=5, backward=True)
        Hn, rstd, mean = G.saved_from_oracle(ctx, G.oracle_forward(ctx, d))
        d["Y"], d["W"] = torch.ldexp(d["Y"], torch.tensor(ey)), torch.ldexp(d["W"], torch.tensor(ew))
        d["R"].zero_()
        want = G.oracle_forward(ctx, d)["Hn"]
        got, gb, ob = G.gpu_forward(ctx, layer, d), G.gpu_backward(ctx, layer, d, Hn, rstd, mean), G.oracle_backward(ctx, d, Hn, rstd, mean)
        out.append([_rel(got["Hn"], want), _rel(gb["dY"], ob["dY"]), _rel(gb["dW"], ob["dW"])])
    for simt, tensor in zip(*out):
        assert tensor < 1.1 * simt


def test_values_that_are_not_finite():
    """An infinite or NaN operand gives what a chain of FMAs gives, also where the other operand's lower parts are zero."""
    t, T, h, ffn, layer = 2, 300, 512, 4096, caat.CAAT_MLP_DOWN
    ctx = G.make_ctx(t, h, ffn, "f32", S=256)
    k = ctx.k_r(layer)
    d = _layer_case(t, T, h, k, "f32", 256, seed=2)
    d["W"] = d["W"].abs().bfloat16().float() + 0.0     # positive, lower parts zero
    d["Y"][0, 7, 11] = float("inf")
    d["Y"][1, 140, 500] = float("nan")
    d["Y"][1, 299, k - 1] = 3.4e38                     # its first part would round to infinity
    d["W"][0, 300, 5] = -float("inf")                  # a private column of rank 0
    got = G.gpu_forward(ctx, layer, d)["Hn"].double().numpy()
    with np.errstate(all="ignore"):
        want = G.oracle_forward(ctx, d)["Hn"].astype(np.float32).astype(np.float64)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    ok = np.isfinite(want)
    assert np.isposinf(got[0, 7, 0]) and np.isnan(got[1, 140, 400]) and np.all(np.abs(got[ok] - want[ok]) <= 1e-4 * np.maximum(np.abs(want[ok]), 1))


def _same_with_infinities(got, want, rel):
    got, want = got.double().numpy(), want.astype(np.float32).astype(np.float64)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isposinf(got), np.isposinf(want))
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    ok = np.isfinite(want)
    assert ((got[ok] - want[ok]) ** 2).sum() ** 0.5 <= rel * (want[ok] ** 2).sum() ** 0.5


@pytest.mark.parametrize("t,T,h,ffn,S", [
    (4, 2000, 768, 3072, 384),      # forward: the shared part over clusters of CTAs; gradients: whole tiles of pairs
    (2, 3000, 1024, 4096, 512),     # whole tiles of pairs, two to six a pair
    (4, 999, 768, 3000, 285),       # element-wise loads; partial tiles of clusters of pairs in forward and weight gradient
    (8, 300, 2048, 5632, 1024),     # more clusters' tiles than clusters
    (2, 6000, 512, 2048, 0),        # weight gradient over clusters of pairs
    (4, 64, 768, 3072, 384),        # data gradient over clusters of pairs; a contraction of one chunk
])
def test_an_infinite_token_and_channel(t, T, h, ffn, S):
    """Whole gradients that are infinite: every tile is computed again, none of the waits around it runs out (the harness reads
    the status), and a weight gradient keeps the sign that a chain gives."""
    layer = caat.CAAT_MLP_DOWN
    ctx = G.make_ctx(t, h, ffn, "f32", S=S)
    d = _layer_case(t, T, h, ctx.k_r(layer), "f32", S, seed=T, backward=True)
    fo = G.oracle_forward(ctx, d)
    Hn, rstd, mean = G.saved_from_oracle(ctx, fo)
    d["Y"][:, T // 2] = float("inf")                   # dW infinite wherever that token has a gradient
    d["W"][0, h - 1] = float("inf")                    # a private channel of rank 0, all of dY[0]
    with np.errstate(all="ignore"):
        ob = G.oracle_backward(ctx, d, Hn, rstd, mean)
    gb = G.gpu_backward(ctx, layer, d, Hn, rstd, mean)
    assert np.isinf(ob["dW"]).all() and np.isinf(ob["dY"][0]).all()
    for name in ("dY", "dW", "dR", "dgamma"):
        _same_with_infinities(gb[name], ob[name], 1e-5)
    d["Y"] = d["Y"].abs()                              # forward: a row of NaN or infinities per rank, a column of infinities
    with np.errstate(all="ignore"):
        fo = G.oracle_forward(ctx, d)
    got = G.gpu_forward(ctx, layer, d)
    assert not np.isfinite(fo["Hn"][0, :, h - 1]).any()
    _same_with_infinities(got["Hn"], fo["Hn"], 1e-5)


CHILD = r"""
import torch
from paper_2506_19645_b200 import caat, synthetic
t, T, h, ffn, layer = 4, 700, 768, 3072, caat.CAAT_MLP_DOWN
ctx = caat.Context(h, ffn, t, 0.5, "f32")
d = synthetic.layer_inputs(t, T, h, ctx.k_r(layer), "f32", seed=1, S=ctx.shared_channels, device="cuda")
mk = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
Hn, X, rstd = mk(t, T, h), mk(t, T, h), mk(t, T)
ws = ctx.alloc_workspace(ctx.workspace_bytes(layer, T, False))
ctx.rowpar_forward(layer, T, d["Y"], d["W"], d["R"], d["gamma"], None, Hn, X, rstd, None, ws)
torch.cuda.synchronize()
print("STATUS", ctx.last_device_status(), ctx.last_device_status(), int(torch.ones(1024, device="cuda").sum().item()))
"""


def test_waits_run_out_and_report_timeout():
    """Stages that are filled but never announced: every role gives up within its poll limit, partial tiles of a cluster included."""
    env = dict(os.environ, CAAT_TC_DEBUG="1024", CAAT_TC_SPINCAP="2048")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    line = [l for l in out.stdout.splitlines() if l.startswith("STATUS")][-1].split()
    assert [int(x) for x in line[1:]] == [caat.CAAT_ETIMEOUT, caat.CAAT_OK, 1024]
