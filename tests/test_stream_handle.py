"""The binding's stream argument on CPU: an explicit stream's handle, torch's raw current stream where
torch offers it, and the public current stream where it does not."""
from types import SimpleNamespace

import torch

from paper_2405_01522_gb300 import rsx


def test_stream_handles(monkeypatch):
    assert rsx._stream(SimpleNamespace(cuda_stream=11)).value == 11
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 2)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=12))
    monkeypatch.setattr(rsx, "_raw_stream", lambda device: 20 + device)
    assert rsx._stream(None).value == 22
    monkeypatch.setattr(rsx, "_raw_stream", None)
    assert rsx._stream(None).value == 12
