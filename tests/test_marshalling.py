"""The binding's stream handle, without a GPU: an explicit stream's own, the
current stream's raw handle, and the documented attribute where torch has no
raw handle to give."""
import types

import pytest
import torch

from paper_2608_06412_gb300 import af


def test_stream_handles(monkeypatch):
    s = types.SimpleNamespace(cuda_stream=77)
    assert af._stream_ptr(s) == 77
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: s)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 100 + d, raising=False)
    assert af._stream_ptr(None) == 103
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert af._stream_ptr(None) == 77


def test_failures_of_the_raw_handle_are_not_hidden(monkeypatch):
    def fail(d):
        raise AttributeError("from inside")
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", fail, raising=False)
    with pytest.raises(AttributeError):
        af._stream_ptr(None)
