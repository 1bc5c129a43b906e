"""The native marshalling rejects what the binding's own checks reject, with their words."""
import pytest
import torch

from paper_2506_19645_b200 import caat


def test_host_tensors_and_non_tensors_are_rejected():
    ctx = caat.Context(256, 1024, 4, 0.5, "bf16")
    y = torch.zeros(4, 8, 256, dtype=torch.bfloat16)
    for bad in (y, 3, "x"):
        with pytest.raises(TypeError, match="Y: expected a CUDA tensor"):
            ctx.rowpar_forward(caat.CAAT_MLP_DOWN, 8, bad, *[None] * 9)
    with pytest.raises(TypeError, match="workspace: expected a CUDA tensor"):
        ctx.block_forward(8, *[None] * 17, workspace=y)


@pytest.mark.gpu
def test_missing_arguments_reach_the_library():
    ctx = caat.Context(256, 1024, 4, 0.5, "bf16")
    for call in (lambda: ctx.rowpar_forward(caat.CAAT_ATTN_OUT, 8, *[None] * 10),
                 lambda: ctx.rowpar_backward(caat.CAAT_ATTN_OUT, 8, *[None] * 14),
                 lambda: ctx.block_backward(8, *[None] * 26), lambda: ctx.colpar_forward(caat.CAAT_ACT_SILU, 64, 8, *[None] * 4)):
        with pytest.raises(caat.CaatError) as e:
            call()
        assert e.value.status == caat.CAAT_EINVAL


@pytest.mark.gpu
def test_device_tensors_of_the_wrong_kind_are_named():
    ctx = caat.Context(256, 1024, 4, 0.5, "bf16")
    ok = torch.zeros(4, 8, 256, dtype=torch.bfloat16, device="cuda")
    for bad, err, text in ((ok.float(), TypeError, "Y: expected torch.bfloat16, got torch.float32"),
                           (ok[:, :4], ValueError, "Y: must be contiguous"),
                           (ok[:2].contiguous(), ValueError, r"Y: expected shape \(4, 8, 256\), got \(2, 8, 256\)")):
        with pytest.raises(err, match=text):
            ctx.rowpar_forward(caat.CAAT_MLP_DOWN, 8, bad, *[None] * 9)
