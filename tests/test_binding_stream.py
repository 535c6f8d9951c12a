"""The stream handed to the library when the caller names none."""
import types

import pytest
import torch

from paper_2404_09531_gb300 import binding


def test_current_stream_without_the_private_name(monkeypatch):
    """A torch that lacks the raw lookup: the public current stream is used."""
    monkeypatch.setattr(binding, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=4321))
    assert binding._stream().value == 4321


def test_given_stream():
    assert binding._stream(types.SimpleNamespace(cuda_stream=77)).value == 77


@pytest.mark.gpu
def test_current_stream_follows_the_context():
    s = torch.cuda.Stream()
    assert (binding._stream().value or 0) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(s):
        assert binding._stream().value == s.cuda_stream
