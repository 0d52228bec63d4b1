"""The binding's stream argument: the current stream's handle with and without
torch's undocumented calls for it, a Stream object's, a number."""

import types

import paper_2608_03473_gb300 as lg


def test_current_stream_without_the_raw_calls(monkeypatch):
    import torch
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.delattr(torch._C, "_cuda_getDevice", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    assert lg._stream_handle(None) == 77


def test_given_streams():
    assert lg._stream_handle(types.SimpleNamespace(cuda_stream=78)) == 78 and lg._stream_handle(79) == 79
