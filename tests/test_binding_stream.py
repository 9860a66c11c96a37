"""The stream a call runs on when none is given: torch's current stream, with and
without torch's private handle call.  No GPU (a stand-in for torch's streams)."""
import types

import pytest


@pytest.mark.parametrize("private_call", [True, False])
@pytest.mark.parametrize("initialized", [True, False])
def test_default_stream(monkeypatch, private_call, initialized):
    import torch
    import paper_2509_16407_gb300 as ws
    t = ws.Table.__new__(ws.Table)
    t.device = 3
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: initialized)
    monkeypatch.setattr(torch.cuda, "is_available", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d: types.SimpleNamespace(cuda_stream=0x1000 + d))
    if private_call:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 0x1000 + d, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert t._stream(None).value == 0x1003
