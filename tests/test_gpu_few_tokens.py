"""Few-token path: shared planes over groups of ranks or k-splits, tiles dealt by length (and round-robin past the table)."""
import pytest

from paper_2506_19645_b200 import caat
from tests import gpu_harness as G
from tests.test_gpu_parity import _check_forward, _layer_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,T,h,ffn,layer,S", [
    (8, 64, 4096, 11008, caat.CAAT_MLP_DOWN, 2048),    # groups of ranks
    (8, 2, 4096, 11008, caat.CAAT_MLP_DOWN, 4096),     # nothing private
    (8, 2, 4096, 11008, caat.CAAT_MLP_DOWN, 0),        # nothing shared
    (6, 33, 768, 3072, caat.CAAT_MLP_DOWN, 383),       # six ranks, odd partition
    (3, 64, 264, 8184, caat.CAAT_MLP_DOWN, 100),       # few tiles: k-splits, a tile of 128 channels mostly empty
    (1, 5, 512, 4096, caat.CAAT_MLP_DOWN, 256),        # one rank
    (2, 1, 16, 16, caat.CAAT_ATTN_OUT, 8),             # K_r = 8: a single k-step
    (16, 3, 16384, 16384, caat.CAAT_ATTN_OUT, 8192),   # more tiles than the dealing table holds
])
def test_few_token_layer(t, T, h, ffn, layer, S):
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S)
    d = _layer_case(t, T, h, ctx.k_r(layer), "bf16", S, seed=T + S)
    _check_forward(ctx, layer, d, "bf16")
