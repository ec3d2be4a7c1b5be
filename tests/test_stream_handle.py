"""The current stream's handle comes through the public torch call where the private one is missing."""
import types

import pytest
import torch


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_without_the_private_call(monkeypatch, missing):
    from paper_1407_4859_gb300.api import _stream_ptr
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 64 + device, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 1, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=4096))
    assert _stream_ptr(None).value == 65
    monkeypatch.delattr(torch._C, missing)
    assert _stream_ptr(None).value == 4096
    assert _stream_ptr(types.SimpleNamespace(cuda_stream=256)).value == 256
