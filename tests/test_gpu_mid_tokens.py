"""Block forward with some hundreds of tokens: both products in one launch with the weights on the row side of a CTA pair's tiles.
Every sum has the bits that the layers give one by one (tokens on the row side), so the new streams are compared bit by bit."""
import pytest
import torch

from paper_2506_19645_b200 import caat, synthetic
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,T,h,ffn,S", [
    (8, 65, 2048, 5632, 1024),      # the fewest tokens, one column tile
    (8, 200, 4096, 11008, 2047),    # an odd partition
    (8, 257, 5120, 13824, 2560),    # a column past one tile
    (8, 300, 4096, 11008, 2048),    # rank groups in fp32 planes
    (8, 300, 4096, 11008, 0),       # nothing shared
    (2, 300, 3072, 8192, 1000),     # shared and private rows end inside a tile
    (8, 511, 2048, 5632, 520),
])
def test_block_forward_has_the_layers_bits(t, T, h, ffn, S):
    _same_bits(t, T, h, ffn, S)


def test_plans_kept_by_shape_serve_their_own_shape():
    """More shapes than plans are kept, each of them twice, the second time in the other order; another partition and another
    set of layers with the same token counts in between."""
    shapes = [(2, T, 1024, 4096, 512) for T in range(65, 129)] + [(2, T, 1024, 4096, 1024) for T in (65, 100, 128)]
    shapes += [(4, T, 1024, 3072, 512) for T in (65, 100, 128)]
    for shape in shapes + shapes[::-1]:
        _same_bits(*shape)


def _same_bits(t, T, h, ffn, S):
    ctx = G.make_ctx(t, h, ffn, "bf16", S=S)
    w = synthetic.Workload("", t, T, h, ffn, S / h, "bf16", "block", False, T + S)
    i = synthetic.block_inputs(w, S, device="cuda")
    mk = lambda *s, dt=torch.bfloat16: torch.empty(*s, dtype=dt, device="cuda")  # noqa: E731
    f32 = torch.float32
    o = {n: mk(t, T, h) for n in ("Hn1", "X1", "Hn2", "X2", "a1", "b1", "a2", "b2")}
    r = [mk(t, T, dt=f32) for _ in range(4)]
    ws = ctx.alloc_workspace(ctx.block_workspace_bytes(T, False))
    ctx.block_forward(T, i["Y_attn"], i["W_o"], i["Y_mlp"], i["W_down"], i["R0"], i["gamma1"], None, i["gamma2"], None, o["Hn1"],
                      o["X1"], r[0], None, o["Hn2"], o["X2"], r[1], None, ws)
    ctx.rowpar_forward(caat.CAAT_ATTN_OUT, T, i["Y_attn"], i["W_o"], i["R0"], i["gamma1"], None, o["a1"], o["b1"], r[2], None, ws)
    ctx.rowpar_forward(caat.CAAT_MLP_DOWN, T, i["Y_mlp"], i["W_down"], o["a1"], i["gamma2"], None, o["a2"], o["b2"], r[3], None, ws)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == caat.CAAT_OK
    assert torch.equal(o["Hn1"], o["a1"]) and torch.equal(o["Hn2"], o["a2"])
    for x, y in ((r[0], r[2]), (r[1], r[3])):
        assert torch.allclose(x, y, rtol=1e-5, atol=0)      # the order of a row's sum of squares differs
