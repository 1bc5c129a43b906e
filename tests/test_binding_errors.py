"""The native marshalling rejects what the binding's own checks reject, with their words."""
import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode

from paper_2506_19645_b200 import caat


def test_host_tensors_and_non_tensors_are_rejected():
    ctx = caat.Context(256, 1024, 4, 0.5, "bf16")
    y = torch.zeros(4, 8, 256, dtype=torch.bfloat16)
    for bad in (y, 3, "x"):
        with pytest.raises(TypeError, match="Y: expected a CUDA tensor"):
            ctx.rowpar_forward(caat.CAAT_MLP_DOWN, 8, bad, *[None] * 9)
    with pytest.raises(TypeError, match="workspace: expected a CUDA tensor"):
        ctx.block_forward(8, *[None] * 17, workspace=y)


def test_tensors_without_storage_raise():
    # inside vmap a tensor has a device but no storage; a fake tensor stands for the CUDA tensor on machines without one
    ctx = caat.Context(256, 1024, 4, 0.5, "bf16")
    args = {"tensor": lambda v: ctx.rowpar_forward(caat.CAAT_MLP_DOWN, 8, v, *[None] * 9),
            "workspace": lambda v: ctx.block_forward(8, *[None] * 17, workspace=v)}
    with FakeTensorMode():
        xs = {"tensor": torch.empty(3, 4, 8, 256, dtype=torch.bfloat16, device="cuda"),
              "workspace": torch.empty(3, 64, dtype=torch.uint8, device="cuda")}
        for name, call in args.items():
            def f(v):
                call(v)
                return v
            with pytest.raises(RuntimeError, match="storage"):
                torch.func.vmap(f)(xs[name])


@pytest.mark.gpu
def test_sparse_tensors_raise():
    ctx = caat.Context(256, 1024, 4, 0.5, "bf16")
    y = torch.zeros(4, 8, 256, dtype=torch.bfloat16, device="cuda").to_sparse()
    with pytest.raises((RuntimeError, ValueError)):
        ctx.rowpar_forward(caat.CAAT_MLP_DOWN, 8, y, *[None] * 9)


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
