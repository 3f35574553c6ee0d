"""The stream that the binding hands to the library is torch's current one, with and without torch's
shortcut to it (no GPU: torch's calls are replaced)."""
import types

import torch

import paper_2009_06628_gb300 as chns


def test_the_stream_is_the_current_one(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=17))
    monkeypatch.setattr(chns, "_raw_stream", lambda device: {3: 17}[device])
    assert chns._stream() == 17
    monkeypatch.setattr(chns, "_raw_stream", None)
    assert chns._stream() == 17
