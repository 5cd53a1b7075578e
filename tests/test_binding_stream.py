"""The stream that a binding call launches on: the one it is given, else the current one, with
torch's raw handle or, where torch has none, with its Stream object."""
import types

import torch

from paper_1802_07210_gb300 import binding as B


def test_stream_handles(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    monkeypatch.setattr(B, "_raw_stream", lambda device: 5000 + device)
    assert B._stream(types.SimpleNamespace(cuda_stream=77)).value == 77
    assert B._stream().value == 5003
    monkeypatch.setattr(B, "_raw_stream", None)
    assert B._stream(types.SimpleNamespace(cuda_stream=77)).value == 77
    assert B._stream().value == 1234
