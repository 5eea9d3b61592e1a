"""The binding's choice of a stream (no GPU needed: torch's functions are replaced)."""
import importlib.util
import os

import torch

from paper_2508_03567_gb300 import binding


class _Stream:
    cuda_stream = 4711


def test_default_stream_without_the_raw_handle_function(monkeypatch):
    """A torch without the private function that returns the raw handle: the public one serves."""
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    spec = importlib.util.spec_from_file_location("binding_without_raw_stream", os.path.abspath(binding.__file__))
    fresh = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(fresh)
    assert fresh._stream_ptr(None) == 4711
    assert fresh._stream_ptr(17) == 17


def test_default_stream_with_the_raw_handle_function(monkeypatch):
    monkeypatch.setattr(binding, "_raw_stream", lambda dev: 100 + dev)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    assert binding._stream_ptr(None) == 103
