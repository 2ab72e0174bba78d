"""The stream of a layer call (CPU): torch's current one on the tensors' device, with
or without torch's private raw-stream function; a device that is not CUDA is refused."""
import types

import pytest
import torch

from paper_2604_08542_gb300 import layer


def test_stream_without_the_raw_function(monkeypatch):
    seen = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d: seen.append(d) or types.SimpleNamespace(cuda_stream=42))
    monkeypatch.setattr(layer, "_raw_stream", None)
    assert layer._stream(torch.device("cuda", 1)) == 42 and seen == [torch.device("cuda", 1)]


def test_stream_with_the_raw_function(monkeypatch):
    monkeypatch.setattr(layer, "_raw_stream", lambda index: 7 + index)
    assert layer._stream(torch.device("cuda", 1)) == 8


def test_a_cpu_device_is_refused():
    with pytest.raises(ValueError, match="cuda device"):
        layer._stream(torch.device("cpu"))
