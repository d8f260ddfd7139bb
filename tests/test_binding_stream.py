"""The binding's stream handle: of the given stream, else the current one, by PyTorch's raw-handle function where this
version has it and by the public call where it has not."""

import types

import pytest

import paper_1701_08547_gb300 as T


def test_given_stream():
    assert T._stream(types.SimpleNamespace(cuda_stream=77)) == 77


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_without_raw_handles(monkeypatch, missing):
    import torch

    monkeypatch.delattr(torch._C, missing, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=123))
    if missing == "_cuda_getDevice":
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 5, raising=False)
    assert T._stream(None) == 123


def test_current_stream_by_raw_handle(monkeypatch):
    import torch

    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 1000 + device, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    assert T._stream(None) == 1003
