"""The binding's default stream, on the CPU: the current stream, with or without the call that torch
keeps for itself (which only saves time)."""
import types

import torch


def test_default_stream_without_the_private_call(pcbp, monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 40 + dev, raising=False)
    assert pcbp._stream(None) == 43
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=77))
    assert pcbp._stream(None) == 77
    assert pcbp._stream(5) == 5
    assert pcbp._stream(types.SimpleNamespace(cuda_stream=9)) == 9
