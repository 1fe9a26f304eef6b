"""CPU: the current stream's handle where torch has no internal accessor for it."""
import types

import torch

from paper_2303_13435_gb300 import api


def test_public_call_stands_in(monkeypatch):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d: types.SimpleNamespace(cuda_stream=100 + d))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(api, "_raw_stream", api._raw_stream_of())
    assert api._stream(None) == 103
    assert api._stream(types.SimpleNamespace(cuda_stream=7)) == 7
