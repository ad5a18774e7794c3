"""The stream that a call without one takes: PyTorch's current stream, by its raw handle where
the PyTorch at hand offers that, else by the public interface."""
from types import SimpleNamespace

import pytest


def test_without_the_raw_handle_call(monkeypatch):
    torch = pytest.importorskip("torch")
    import paper_1810_08860_gb300 as lfm

    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=0x1230))
    assert lfm._stream_handle(None).value == 0x1230
    assert lfm._stream_handle(SimpleNamespace(cuda_stream=0x4560)).value == 0x4560


def test_with_the_raw_handle_call(monkeypatch):
    torch = pytest.importorskip("torch")
    import paper_1810_08860_gb300 as lfm

    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 0x7000 + device, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    assert lfm._stream_handle(None).value == 0x7003
