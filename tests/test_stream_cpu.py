"""The stream handle that the binding passes: a given stream's, else torch's current one, with or
without torch's non-public shortcut to its handle."""
import types

import torch

import paper_1708_09689_gb300 as pv


def test_the_current_stream_is_found_without_the_shortcut(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=0x1230))
    monkeypatch.setattr(pv, "_raw_stream", None)
    assert pv._stream().value == 0x1230
    assert pv._stream(types.SimpleNamespace(cuda_stream=0x4560)).value == 0x4560


def test_the_shortcut_asks_for_the_current_device(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(pv, "_raw_stream", lambda device: 0x1000 + device)
    assert pv._stream().value == 0x1003
