"""The binding's current stream, with torch's raw-handle functions and in a torch that does not have them."""
import types

import pytest
import torch

from paper_2606_01009_gb300 import melt


@pytest.fixture
def cuda(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=77))
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 100 + d, raising=False)
    return monkeypatch


def test_raw_handle(cuda):
    assert melt._stream_ptr(None) == 103


@pytest.mark.parametrize("name", ["_cuda_getDevice", "_cuda_getCurrentRawStream"])
def test_torch_without_raw_handles(cuda, name):
    cuda.delattr(torch._C, name)
    assert melt._stream_ptr(None) == 77


def test_given_streams(cuda):
    assert melt._stream_ptr(5) == 5
    assert melt._stream_ptr(types.SimpleNamespace(cuda_stream=9)) == 9
