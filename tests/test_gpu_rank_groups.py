"""Forward with few row tiles: the shared columns' rank loop split into groups of ranks (fp32 planes and their sum)."""
import numpy as np
import pytest
import torch

from paper_2506_19645_b200 import caat, synthetic
from tests import gpu_harness as G
from tests.helpers import f64
from tests.test_gpu_parity import _check_forward, _layer_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,T,h,ffn,layer,S,norm", [
    (8, 65, 4096, 11008, caat.CAAT_MLP_DOWN, 2048, 0),     # one row tile, a group per rank
    (8, 300, 4096, 11008, caat.CAAT_MLP_DOWN, 4096, 0),    # everything shared
    (8, 257, 2048, 5632, caat.CAAT_ATTN_OUT, 1433, 1),     # ragged row tile, partition off the 8-channel grid
    (6, 130, 768, 3072, caat.CAAT_MLP_DOWN, 5, 0),         # six ranks (groups of 3 and 2), almost nothing shared
    (3, 100, 768, 3072, caat.CAAT_MLP_DOWN, 761, 0),       # three ranks: a ragged last group
    (8, 1000, 4096, 11008, caat.CAAT_MLP_DOWN, 2048, 0),   # room for four planes only
])
def test_forward_with_few_row_tiles(t, T, h, ffn, layer, S, norm):
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S, norm=norm)
    d = _layer_case(t, T, h, ctx.k_r(layer), "bf16", S, seed=T + S)
    _check_forward(ctx, layer, d, "bf16")


@pytest.mark.parametrize("t,S", [(8, 256), (4, 100), (8, 512)])
def test_rank_groups_are_exact_on_integers(t, S):
    T, h, K_r = 90, 512, 128
    Y = synthetic.small_integers((t, T, K_r), -2, 2, seed=S)
    W = synthetic.small_integers((t, h, K_r), 0, 1, seed=S + 1)
    R = synthetic.small_integers((t, T, h), -8, 8, seed=S + 2)
    W[:, :, 16:] = 0        # sums stay below 256: exact in bf16
    d = {"Y": Y, "W": W, "R": R, "gamma": torch.ones(h).bfloat16(), "beta": None}
    ctx = G.make_ctx(t, h, t * K_r, "bf16", S=S, alpha=1.0)
    assert np.array_equal(f64(G.gpu_forward(ctx, caat.CAAT_MLP_DOWN, d)["Hn"]), G.oracle_forward(ctx, d)["Hn"])


@pytest.mark.parametrize("t,T,h,dtype", [
    (8, 300, 4096, "bf16"),     # just over one token per CTA: every CTA starts and stops inside a token
    (8, 3, 2048, "bf16"),       # fewer units than CTAs
    (4, 70, 768, "bf16"),       # warp-per-token kernel, ragged last group
    (8, 450, 1024, "f32"),      # two token rows per CTA
])
@pytest.mark.parametrize("norm", [0, 1])
def test_forward_rows_with_units_dealt_inside_tokens(t, T, h, dtype, norm):
    ctx = G.make_ctx(t, h, h, dtype, S=h // 2, norm=norm, no_decode=True)
    d = _layer_case(t, T, h, ctx.k_r(caat.CAAT_ATTN_OUT), dtype, h // 2, seed=T)
    _check_forward(ctx, caat.CAAT_ATTN_OUT, d, dtype)


def test_compact_stream_in_place_with_few_tokens():
    t, T, h, S = 8, 300, 2048, 1024
    ctx = G.make_ctx(t, h, 4096, "bf16", S=S)
    d = _layer_case(t, T, h, 512, "bf16", S, seed=1)
    dev = {k: v.cuda() for k, v in d.items()}
    Rs, Rp = dev["R"][0, :, :S].contiguous(), dev["R"][:, :, S:].contiguous()
    ws = ctx.alloc_workspace(ctx.workspace_bytes(caat.CAAT_MLP_DOWN, T, False))
    out = []
    for in_place in (False, True):
        a, b = (Rs.clone(), Rp.clone()) if in_place else (torch.empty_like(Rs), torch.empty_like(Rp))
        X, rstd = torch.empty_like(dev["R"]), torch.empty(t, T, device="cuda")
        ctx.rowpar_forward_compact(caat.CAAT_MLP_DOWN, T, dev["Y"], dev["W"], a if in_place else Rs, b if in_place else Rp,
                                   dev["gamma"], None, a, b, X, rstd, None, ws)
        torch.cuda.synchronize()
        out.append((a, b, X, rstd))
    assert all(torch.equal(x, y) for x, y in zip(*out))
