"""Whose stream the binding takes (api._stream_handle): a tensor's own device's; a tensor
without one is refused, as torch.cuda.current_stream refuses its device."""
import pytest
import torch

from paper_2512_10059_gb300 import api


def test_a_host_tensor_has_no_stream(monkeypatch):
    asked = []
    monkeypatch.setattr(api, "_raw_stream", lambda dev: asked.append(dev) or 0)
    with pytest.raises(ValueError):
        api._stream_handle(torch.zeros(256, dtype=torch.uint8))
    with pytest.raises(ValueError):  # before any copy from its address
        api.ragged_status(torch.zeros(256, dtype=torch.uint8))
    assert asked == []


def test_a_given_stream_is_taken():
    class S:
        cuda_stream = 77
    assert api._stream_handle(torch.zeros(1), S()) == 77
