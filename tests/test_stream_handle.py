"""Stream handles of the Python calls, also with a torch that lacks the private fast path (no GPU:
the torch calls are stand-ins)."""
from types import SimpleNamespace

import torch

from paper_2410_21888_gb300 import rimp2


def test_handles(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=77))
    assert rimp2._stream_handle(SimpleNamespace(cuda_stream=5)) == 5
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 100 + d, raising=False)
    assert rimp2._stream_handle(None) == 103
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert rimp2._stream_handle(None) == 77
