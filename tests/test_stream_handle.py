"""The stream handle that the binding passes: torch's current stream, with and without
torch's private accessors."""
import types

import pytest
import torch

from paper_2606_31160_gb300 import sd


@pytest.mark.parametrize("name", ["_raw_stream", "_raw_device"])
def test_without_the_private_accessor(monkeypatch, name):
    monkeypatch.setattr(sd, name, None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    assert sd._stream() == 1234


@pytest.mark.gpu
def test_both_ways_name_the_current_stream(monkeypatch):
    side = torch.cuda.Stream()
    for stream in (torch.cuda.current_stream(), side):
        with torch.cuda.stream(stream):
            fast = sd._stream()
            with monkeypatch.context() as m:
                m.setattr(sd, "_raw_stream", None)
                assert sd._stream() == fast == stream.cuda_stream
