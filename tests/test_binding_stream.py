"""The stream a call of the binding runs on when none is given, on the host."""
import types

import torch

from paper_2609_24294_gb300 import zfpx as z


def test_current_stream_by_handle_and_by_object(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=0x30))
    monkeypatch.setattr(z, "_raw_stream", lambda device: 0x10 * device)
    assert z._stream(None).value == 0x30
    # a PyTorch without the raw handle
    monkeypatch.setattr(z, "_raw_stream", None)
    assert z._stream(None).value == 0x30
    assert z._stream(types.SimpleNamespace(cuda_stream=0x50)).value == 0x50
