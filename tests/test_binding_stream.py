"""CPU tests of the stream argument that the torch convenience passes on: a stream's own handle, the
current stream's raw handle, and the current stream object's where torch has no raw handle."""
import types

import pytest


@pytest.fixture
def torch_cuda(monkeypatch):
    import torch
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    return torch


def test_given_stream():
    from paper_2512_15187_gb300 import binding
    assert binding._stream(types.SimpleNamespace(cuda_stream=1 << 40)) == 1 << 40


def test_current_stream(torch_cuda, monkeypatch):
    from paper_2512_15187_gb300 import binding
    monkeypatch.setattr(torch_cuda._C, "_cuda_getCurrentRawStream", lambda dev: 100 + dev, raising=False)
    assert binding._stream(None) == 103


def test_current_stream_without_torchs_raw_handle(torch_cuda, monkeypatch):
    from paper_2512_15187_gb300 import binding
    monkeypatch.delattr(torch_cuda._C, "_cuda_getCurrentRawStream", raising=False)
    assert binding._stream(None) == 77
