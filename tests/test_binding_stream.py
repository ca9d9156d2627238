"""Which stream the binding hands to the library, without a GPU."""
import types

import torch


def test_current_stream_without_the_private_call(monkeypatch):
    """A torch without the raw-stream call serves through its public one."""
    from paper_2505_18932_gb300 import gvs
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(gvs, "_raw_stream", None, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=0x1230))
    assert gvs._stream(None).value == 0x1230
    assert gvs._stream(types.SimpleNamespace(cuda_stream=0x4560)).value == 0x4560
