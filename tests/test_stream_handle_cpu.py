"""The current stream's handle comes from PyTorch's private call where there is one and
from the public API otherwise."""
import types

import torch

from paper_1204_4302_gb300 import plan


def test_handle_without_the_private_call(monkeypatch):
    asked = []

    def current_stream(index):
        asked.append(index)
        return types.SimpleNamespace(cuda_stream=77)
    monkeypatch.setattr(torch.cuda, "current_stream", current_stream)
    assert plan._stream_getter(types.SimpleNamespace())(3) == 77 and asked == [3]


def test_handle_by_the_private_call():
    c = types.SimpleNamespace(_cuda_getCurrentRawStream=lambda index: 10 + index)
    assert plan._stream_getter(c)(2) == 12
