"""The handle of torch's current stream, with and without torch's private shortcut to it."""
import types

import pytest

import paper_1803_08601_gb300 as pkg


@pytest.mark.parametrize("missing", [(), ("_cuda_getCurrentRawStream",), ("_cuda_getDevice",)])
@pytest.mark.parametrize("initialized", [True, False])
def test_current_stream_without_the_private_names(monkeypatch, missing, initialized):
    torch = pytest.importorskip("torch")
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: initialized)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=7))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 11 + device, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 2, raising=False)
    for name in missing:
        monkeypatch.delattr(torch._C, name)
    assert pkg._stream_handle() == (13 if initialized and not missing else 7)
    assert pkg._stream_handle(types.SimpleNamespace(cuda_stream=5)) == 5
