"""Which stream a call without one goes to (no GPU: PyTorch's lookups are
replaced)."""
import types

import torch

from paper_1112_0065_gb300.dedisp import _stream_handle


def test_current_stream_with_and_without_the_raw_lookup(monkeypatch):
    """The current device's current stream, through PyTorch's raw lookup where
    the build has it and through the public Stream object where it has not; a
    given stream is taken as it is."""
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 1000 + device, raising=False)
    assert _stream_handle(None) == 1003
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert _stream_handle(None) == 77
    assert _stream_handle(types.SimpleNamespace(cuda_stream=5)) == 5
