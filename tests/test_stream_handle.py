"""The stream a call runs on: the caller's, or torch's current one, with torch's
quick way to its handle and without it."""
import torch

from paper_2604_21749_gb300 import api


class _Stream:
    cuda_stream = 4711


def test_the_callers_stream():
    assert api._stream(_Stream()) == 4711


def test_the_current_stream(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream())
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.delattr(torch._C, name, raising=False)
    assert api._stream() == 4711
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    assert api._stream() == 4711
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 100 + device, raising=False)
    assert api._stream() == 103
