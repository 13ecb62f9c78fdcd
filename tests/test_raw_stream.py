"""CubeModel's stream argument without a GPU: the stream's own handle, torch's raw handle
of the device's current stream where torch has the call, and else the current stream
object's."""
import types

import pytest
import torch

model = pytest.importorskip("paper_2412_08265_gb300.model")


def test_raw_stream(monkeypatch):
    dev = torch.device("cuda", 3)
    assert model._raw_stream(types.SimpleNamespace(cuda_stream=77), dev) == 77
    monkeypatch.setattr(model, "_current_raw_stream", lambda index: 100 + index)
    assert model._raw_stream(None, dev) == 103
    monkeypatch.setattr(model, "_current_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d: types.SimpleNamespace(cuda_stream=200 + d.index))
    assert model._raw_stream(None, dev) == 203
