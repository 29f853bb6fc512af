"""The default stream argument: the current stream's handle, from torch's private
call where it exists and from the public one where it does not."""
import types

import torch

import paper_2609_36835_gb300 as pk


def test_current_stream_with_and_without_the_private_call(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=22))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 11 + dev, raising=False)
    assert pk._stream_handle(None) == 14
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert pk._stream_handle(None) == 22
    assert pk._stream_handle(7) == 7 and pk._stream_handle(types.SimpleNamespace(cuda_stream=9)) == 9
