"""The binding's default stream where torch lacks the call for the raw handle (no GPU:
the public call is a stand-in)."""
from types import SimpleNamespace

from gpu_common import load_pkg


def test_public_call_stands_in(monkeypatch):
    import torch
    sp = load_pkg()
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=4242))
    assert sp._stream(None).value == 4242
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 17 + device,
                        raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 1)
    assert sp._stream(None).value == 18
