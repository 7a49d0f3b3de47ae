"""The binding's stream handle without a GPU: a stream given, the current one
by torch's raw call, and by a Stream object where torch has no raw call."""
import types

import torch


def test_raw_stream_with_and_without_torchs_raw_call(monkeypatch):
    from paper_1402_7216_gb300 import _raw_stream
    assert _raw_stream(types.SimpleNamespace(cuda_stream=7)) == 7
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 100 + device, raising=False)
    assert _raw_stream(None) == 103
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=11))
    assert _raw_stream(None) == 11
