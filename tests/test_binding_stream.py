"""The current stream's handle, with and without torch's functions that read it directly."""
import types

import torch

from paper_2503_23186_b200 import binding


def test_public_call_where_the_direct_one_is_missing(monkeypatch):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    assert binding._stream() == 1234


def test_direct_call(monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 100 + device, raising=False)
    assert binding._stream() == 103
