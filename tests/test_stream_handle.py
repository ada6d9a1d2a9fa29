"""The stream a binding call uses when the caller names none, with no GPU: torch's
current stream, also on a torch without the private functions that give its
handle directly."""
import types

import pytest
import torch

import paper_2605_06892_gb300 as hsa


@pytest.mark.parametrize("missing", ["_raw_stream", "_current_device"])
def test_current_stream_without_the_private_functions(monkeypatch, missing):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda: types.SimpleNamespace(cuda_stream=4711))
    monkeypatch.setattr(hsa, "_raw_stream", lambda device: 1)
    monkeypatch.setattr(hsa, "_current_device", lambda: 0)
    monkeypatch.setattr(hsa, missing, None)
    assert hsa._stream(None) == 4711


def test_named_streams_are_taken_as_they_are():
    assert hsa._stream(12) == 12
    assert hsa._stream(types.SimpleNamespace(cuda_stream=34)) == 34
