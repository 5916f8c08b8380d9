"""The current stream's handle with and without torch's direct accessor (CPU)."""

import types

import pytest

torch = pytest.importorskip("torch")

import paper_1409_2014_gb300 as pkg  # noqa: E402


def test_stream_handle(monkeypatch):
    dev = torch.device("cuda", 1)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 100 + index, raising=False)
    assert pkg._raw_stream(dev) == 101
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device: types.SimpleNamespace(cuda_stream=200 + device.index))
    assert pkg._raw_stream(dev) == 201
