"""The current stream's handle comes from PyTorch's internal raw call where there is one, and from the public
Stream object where there is not (PyTorch keeps no promise about the former)."""
import types

import torch

from paper_1301_0514_gb300 import _lib


def test_stream_handle_without_the_raw_call(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.delattr(torch._C, name, raising=False)
    assert _lib._stream(None) == 1234


def test_stream_handle_of_an_explicit_stream():
    assert _lib._stream(types.SimpleNamespace(cuda_stream=77)) == 77
    assert _lib._stream(5) == 5
