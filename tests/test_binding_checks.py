"""What the binding refuses before the library, which sees bare pointers, is called.  Nothing here needs a GPU."""
import importlib.util
import types

import pytest
import torch

import paper_2510_00236_b200 as pe
from paper_2510_00236_b200 import binding

BF16 = torch.bfloat16


# x 2 x 3 x 9 x 8 under a 3 x 3 kernel, stride (2, 1), padding (1, 0), dilation (1, 2): 5 x 4 positions
@pytest.mark.parametrize("shape,device", [((2, 4, 5, 3), "cpu"), ((2, 4, 4, 4), "cpu"), ((1, 4, 5, 4), "cpu"), ((2, 4, 4, 5), "cpu"),
                                          ((2, 4, 6, 4), "cpu"), ((2, 4, 5, 4), "meta")])
def test_convolution_refuses_cotangents_of_another_size_or_device(shape, device):
    x, grad_out = torch.zeros((2, 3, 9, 8), dtype=BF16), torch.zeros(shape, dtype=BF16, device=device)
    mean, stat = torch.zeros((4, 27)), torch.zeros((4, 27))
    with pytest.raises(ValueError, match="grad_out"):
        pe.pe_conv2d_stats(x, grad_out, (3, 3), "square", (2, 1), (1, 0), (1, 2), mean, stat)


def test_convolution_of_the_right_size_reaches_the_library():
    x, grad_out = torch.zeros((2, 3, 9, 8), dtype=BF16), torch.zeros((2, 4, 5, 4), dtype=BF16)
    mean, stat = torch.zeros((4, 27)), torch.zeros((4, 27))
    with pytest.raises(pe.PestatsError):            # a tensor on the CPU
        pe.pe_conv2d_stats(x, grad_out, (3, 3), "square", (2, 1), (1, 0), (1, 2), mean, stat)


@pytest.mark.parametrize("workspace", [torch.empty(4096, dtype=torch.uint8, device="meta"), torch.zeros(1, dtype=torch.uint8).expand(1 << 20),
                                       torch.zeros(8192, dtype=torch.uint8)[::2]])
def test_padded_call_refuses_a_workspace_the_kernels_cannot_write(workspace):
    X, out = torch.zeros((2, 4, 9), dtype=BF16), torch.zeros((9, 9))
    with pytest.raises(ValueError, match="workspace"):
        pe.pe_linear_stats_padded(X, X, "square", 0, out, torch.zeros((9, 9)), None, workspace)


def test_lookups_without_torch_private_functions(monkeypatch):
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.delattr(torch._C, name, raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda dev: types.SimpleNamespace(cuda_stream=1000 + dev))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    spec = importlib.util.spec_from_file_location("paper_2510_00236_b200.binding_again", binding.__file__)
    again = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(again)
    assert again._raw_stream(2) == 1002 and again._current_device() == 3


@pytest.mark.parametrize("phi,mean,stat,sign,copies", [("square", 1, 1, 1, 4), ("square", 1, 1, 0, 3), ("square", 0, 1, 0, 2), ("sign", 1, 1, 0, 2),
                                                       ("sign", 0, 1, 0, 1), ("identity", 1, 1, 0, 0), ("identity", 0, 1, 0, 0), ("square", 1, 0, 0, 0)])
def test_one_token_workspace_follows_the_outputs(phi, mean, stat, sign, copies):
    B, d_in, d_out = 4096, 512, 1024
    one = 2 * B * (d_in + d_out)
    need = pe.pe_linear_stats_padded_workspace_bytes_for(B, 1, d_in, d_out, phi, mean, stat, sign)
    assert copies * one <= need <= copies * (one + 2 * B)       # beside the copies: a few bytes per example
    assert need <= pe.pe_linear_stats_padded_workspace_bytes(B, 1, d_in, d_out)
    if copies == 0:             # widths that TMA cannot address need a copy for the mean too
        assert pe.pe_linear_stats_padded_workspace_bytes_for(B, 1, 513, d_out, phi, mean, stat, sign) >= 2 * B * (513 + d_out)


class _NoMemory(torch.Tensor):
    def new_empty(self, size, dtype=None, **kw):
        if dtype == torch.uint8:
            raise torch.OutOfMemoryError("no memory for a workspace")
        return super().new_empty(size, dtype=dtype, **kw)


# single tokens, and a width that is no multiple of 8
@pytest.mark.parametrize("B,T,d_in,d_out", [(128, 1, 1024, 1024), (64, 8, 513, 512)])
def test_calls_without_memory_for_a_workspace_are_the_ordinary_ones(monkeypatch, B, T, d_in, d_out):
    X, dY = (torch.zeros((B, T, d), dtype=BF16).as_subclass(_NoMemory) for d in (d_in, d_out))
    outs = [torch.empty((d_out, d_in)) for _ in range(3)]
    assert pe.pe_linear_stats_padded_workspace_bytes(B, T, d_in, d_out) > 0
    called = []
    monkeypatch.setattr(binding, "_launch", lambda name, *args: called.append(name))
    pe.pe_linear_stats(X, dY, "square", outs[0], outs[1])
    pe.pe_linear_stats_accumulate(X, dY, "sign", outs[0], outs[1])
    pe.pe_linear_stats_all(X, dY, *outs)
    assert called == ["pe_linear_stats", "pe_linear_stats_accumulate", "pe_linear_stats_all"]
