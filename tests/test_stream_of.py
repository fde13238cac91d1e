"""The stream that the convenience wrapper hands to the library, with and
without torch's function for the raw stream."""
import types

import torch

from paper_2603_20966_gb300 import sketch


def test_stream_without_the_raw_stream_function(monkeypatch):
    A = torch.zeros(1)
    monkeypatch.setattr(sketch, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda device: types.SimpleNamespace(cuda_stream=(device, 77)))
    assert sketch._stream_of(A) == (A.device, 77)
    monkeypatch.setattr(sketch, "_raw_stream", lambda index: 100 + index)
    assert sketch._stream_of(A) == 100 + A.get_device()
