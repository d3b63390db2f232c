"""The current stream's handle where torch has no raw accessor (no GPU)."""
import types

import torch

from paper_2403_16862_gb300 import api


def test_stream_without_the_raw_accessor(monkeypatch):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=77))
    assert api._stream() == 77


def test_stream_with_the_raw_accessor(monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 100 + device, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    assert api._stream() == 103
