"""The current stream's handle comes through the public torch call where the private one is missing."""
import types

import pytest
import torch


@pytest.mark.parametrize("missing", ["_RAW_STREAM", "_RAW_DEVICE"])
def test_current_stream_without_the_private_call(monkeypatch, missing):
    from paper_1407_4859_gb300 import api
    monkeypatch.setattr(api, "_RAW_STREAM", lambda device: 64 + device)
    monkeypatch.setattr(api, "_RAW_DEVICE", lambda: 1)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=4096))
    assert api._stream_ptr(None).value == 65
    monkeypatch.setattr(api, missing, None)
    assert api._stream_ptr(None).value == 4096
    assert api._stream_ptr(types.SimpleNamespace(cuda_stream=256)).value == 256
