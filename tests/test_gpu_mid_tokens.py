"""Block forward with some hundreds of tokens: both products in one launch with the weights on the row side of a CTA pair's tiles.
Every sum has the bits that the layers give one by one (tokens on the row side), so the new streams are compared bit by bit.  That
the form is the one that runs is read from the launches' own report in a child process."""
import os
import re
import subprocess
import sys

import pytest
import torch

from paper_2506_19645_b200 import caat, synthetic
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu

CASES = [   # t, T, h, ffn, S, norm, compact
    (8, 65, 2048, 5632, 1024, 0, False),      # the fewest tokens, one column tile
    (8, 200, 4096, 11008, 2047, 0, False),    # an odd partition
    (8, 257, 5120, 13824, 2560, 0, False),    # a column past one tile
    (8, 300, 4096, 11008, 2048, 0, False),    # rank groups in fp32 planes
    (8, 300, 4096, 11008, 0, 0, False),       # nothing shared
    (2, 160, 3072, 8192, 1500, 0, False),     # two ranks; shared and private rows end inside a tile
    (2, 511, 3072, 8192, 2304, 0, False),     # the widest tile, two of them, the last column beside the tokens
    (2, 512, 3072, 8192, 2304, 0, False),     # the most tokens
    (4, 400, 1536, 6144, 1536, 0, False),     # nothing private
    (2, 160, 1024, 4096, 512, 1, False),      # LayerNorm
    (4, 300, 1536, 6144, 768, 0, True),       # the stream that stores its shared channels once
    (2, 128, 1024, 4096, 512, 1, True),
]


def _mk(*shape, dt=torch.bfloat16):
    return torch.empty(*shape, dtype=dt, device="cuda")


class Block:
    def __init__(self, t, T, h, ffn, S, norm=0, compact=False):
        self.t, self.T, self.h, self.S, self.norm, self.compact = t, T, h, S, norm, compact
        self.ctx = G.make_ctx(t, h, ffn, "bf16", S=S, norm=norm)
        self.i = synthetic.block_inputs(synthetic.Workload("", t, T, h, ffn, S / h, "bf16", "block", False, T + S), S, device="cuda")
        ramp = torch.linspace(-0.2, 0.2, h, device="cuda").bfloat16()
        self.i.update(gamma1=1 + ramp, gamma2=1 - ramp, beta1=ramp if norm else None, beta2=-ramp if norm else None)
        self.ws = self.ctx.alloc_workspace(self.ctx.block_workspace_bytes(T, False))
        self.out, self.stats = self.outputs(compact)

    def outputs(self, compact):
        t, T, h, S = self.t, self.T, self.h, self.S
        layer = lambda: [*((_mk(T, S), _mk(t, T, h - S)) if compact else (_mk(t, T, h),)), _mk(t, T, h)]  # noqa: E731
        return layer() + layer(), [_mk(t, T, dt=torch.float32) for _ in range(4)]

    def R0(self):
        R = self.i["R0"]
        return (R[0, :, :self.S].contiguous(), R[:, :, self.S:].contiguous()) if self.compact else (R,)

    def block(self, R0):
        i, n = self.i, len(R0) + 1
        m = self.stats[2:] if self.norm else [None, None]
        f = self.ctx.block_forward_compact if self.compact else self.ctx.block_forward
        f(self.T, i["Y_attn"], i["W_o"], i["Y_mlp"], i["W_down"], *R0, i["gamma1"], i["beta1"], i["gamma2"], i["beta2"], *self.out[:n],
          self.stats[0], m[0], *self.out[n:], self.stats[1], m[1], self.ws)

    def layers(self):
        """The layers one by one on the stream that every rank holds, in the layout of the block's outputs."""
        (out, r), i, T, S = self.outputs(False), self.i, self.T, self.S
        m = r[2:] if self.norm else [None, None]
        self.ctx.rowpar_forward(caat.CAAT_ATTN_OUT, T, i["Y_attn"], i["W_o"], i["R0"], i["gamma1"], i["beta1"], out[0], out[1], r[0], m[0],
                                self.ws)
        self.ctx.rowpar_forward(caat.CAAT_MLP_DOWN, T, i["Y_mlp"], i["W_down"], out[0], i["gamma2"], i["beta2"], out[2], out[3], r[1], m[1],
                                self.ws)
        if self.compact:
            out = [out[0][0, :, :S], out[0][:, :, S:], out[1], out[2][0, :, :S], out[2][:, :, S:], out[3]]
        return out, r

    def check(self):
        want, r = self.layers()
        torch.cuda.synchronize()
        assert self.ctx.last_device_status() == caat.CAAT_OK
        n = len(self.out) // 2
        for k, (x, y) in enumerate(zip(self.out, want)):
            # the order of a row's sums of squares differs, and with it the last bit of a normalised value
            if k % n == n - 1:
                assert torch.allclose(x.float(), y.float(), rtol=2 ** -7, atol=2 ** -8)
            else:
                assert torch.equal(x, y)
        for x, y in zip(self.stats[:2], r[:2]):
            assert torch.allclose(x, y, rtol=1e-5, atol=0)


@pytest.mark.parametrize("t,T,h,ffn,S,norm,compact", CASES)
def test_block_forward_has_the_layers_bits(t, T, h, ffn, S, norm, compact):
    b = Block(t, T, h, ffn, S, norm, compact)
    b.block(b.R0())
    b.check()


def test_replayed_from_a_graph_on_other_inputs():
    b = Block(8, 300, 2048, 5632, 1024)
    R0 = b.R0()
    b.block(R0)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        b.block(R0)
    for k in range(2):
        for name in ("Y_attn", "Y_mlp", "W_down"):
            b.i[name].copy_(b.i[name].flip(0))
        g.replay()
        b.check()


CHILD = r"""
import sys
import torch
from tests.test_gpu_mid_tokens import CASES, Block
for case in CASES:
    b = Block(*case)
    torch.cuda.synchronize()
    print("CASE", *case, file=sys.stderr, flush=True)
    b.block(b.R0())
    torch.cuda.synchronize()
"""


def test_the_cases_take_the_form_that_they_are_for():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, CAAT_TC_VERBOSE="1", PYTHONPATH=root)
    out = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    runs = out.stderr.split("CASE ")[1:]
    assert len(runs) == len(CASES)
    for case, text in zip(CASES, runs):
        t, T, h, ffn, S = case[:5]
        launches = re.findall(r"BN=(\d+) cg=(\d+) .*r0 M=(\d+) N=(\d+)", text)
        assert len(launches) == 1, (case, text)                    # both layers in one launch
        bn, cg, rows, cols = map(int, launches[0])
        assert cg == 2 and cols == T and rows == (S or h), (case, text)      # channels on the rows, tokens on the columns
        assert bn == (T + -(-T // 256) - 1) // -(-T // 256) + 31 & ~31


def test_plans_kept_by_shape_serve_their_own_shape():
    """More shapes than plans are kept, each of them twice, the second time in the other order; another partition and another
    set of layers with the same token counts in between."""
    shapes = [(2, T, 1024, 4096, 512) for T in range(65, 129)] + [(2, T, 1024, 4096, 1024) for T in (65, 100, 128)]
    shapes += [(4, T, 1024, 3072, 512) for T in (65, 100, 128)]
    for shape in shapes + shapes[::-1]:
        b = Block(*shape)
        b.block(b.R0())
        b.check()
