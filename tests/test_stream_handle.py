"""The binding's stream handle does not depend on a private call of torch being there."""
import torch

from paper_2205_12268_b200 import wcc


def test_without_the_private_call(monkeypatch):
    class Stream:
        cuda_stream = 17

    monkeypatch.setattr(wcc, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: Stream)
    assert wcc._stream() == 17
