"""CUDA-core GEMM: both kernels (128 x 64 tiles of a CTA; 32 x 32 tiles with the contraction split over warps and a cluster), the
three operand layouts, 16-byte and element-wise loads, at the edges of tiles and of the split."""
import pytest

from paper_2506_19645_b200 import caat
from tests import gpu_harness as G
from tests.test_gpu_parity import _check_backward, _check_forward, _layer_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,T,h,ffn,layer,S,dtype", [
    (2, 128, 256, 1024, caat.CAAT_MLP_DOWN, 128, "f32"),     # warp tiles, clusters
    (2, 1, 8, 16, caat.CAAT_MLP_DOWN, 4, "f32"),             # a single element per product row
    (8, 33, 8, 8, caat.CAAT_ATTN_OUT, 8, "f32"),             # K_r = 1: a stride of one on both axes
    (2, 31, 40, 66, caat.CAAT_MLP_DOWN, 17, "f32"),          # K_r = 33 and an odd partition: no 16-byte loads
    (3, 65, 264, 300, caat.CAAT_MLP_DOWN, 100, "f32"),       # K_r = 100: 16-byte loads, remainders on every axis
    (4, 1000, 768, 1000, caat.CAAT_MLP_DOWN, 384, "f32"),    # CTA tiles in the backward, K_r = 250: element-wise loads
    (4, 999, 768, 3072, caat.CAAT_ATTN_OUT, 388, "f32"),     # CTA tiles in the backward, 16-byte loads, remainders on rows and columns
    (2, 777, 1032, 1032, caat.CAAT_ATTN_OUT, 1032, "f32"),   # everything shared: long contraction split over clusters
    (2, 777, 1032, 1032, caat.CAAT_ATTN_OUT, 0, "f32"),      # nothing shared
    (2, 90, 256, 1028, caat.CAAT_MLP_DOWN, 128, "bf16"),     # bf16 with K_r = 514: warp tiles
    (4, 700, 768, 3000, caat.CAAT_MLP_DOWN, 100, "bf16"),    # bf16 with K_r = 750: CTA tiles in the backward
])
def test_cuda_core_layer(t, T, h, ffn, layer, S, dtype):
    ctx = G.make_ctx(t, h, ffn, dtype, S=S)
    d = _layer_case(t, T, h, ctx.k_r(layer), dtype, S, seed=T + S, backward=True)
    _check_forward(ctx, layer, d, dtype)
    _check_backward(ctx, layer, d, dtype)
