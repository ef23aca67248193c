"""The stream a call runs on: the current one by torch's private query, or by its public one where a
torch has no other; or the one that is given.  CPU only."""
import importlib.util
from types import SimpleNamespace

import torch

from paper_2608_20172_gb300 import binding


def test_current_stream_without_the_private_query(monkeypatch):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    fresh = importlib.util.module_from_spec(importlib.util.find_spec(binding.__name__))
    fresh.__spec__.loader.exec_module(fresh)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=77))
    assert fresh._stream(None) == 77


def test_current_and_given_streams(monkeypatch):
    monkeypatch.setattr(binding, "_raw_stream", lambda device: 100 + device)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    assert binding._stream(None) == 103
    assert binding._stream(SimpleNamespace(cuda_stream=5)) == 5
    assert binding._stream(6) == 6
