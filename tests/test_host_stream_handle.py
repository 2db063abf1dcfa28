"""The handle of the current stream, with and without PyTorch's private names for it."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib  # noqa: E402


@pytest.mark.parametrize("initialised", [False, True])
@pytest.mark.parametrize("missing", [(), ("_cuda_getCurrentRawStream",), ("_cuda_getDevice",),
                                     ("_cuda_getCurrentRawStream", "_cuda_getDevice")])
def test_current_stream_handle(monkeypatch, initialised, missing):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: initialised)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=77))
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 70 + device, raising=False)
    for name in missing:
        monkeypatch.delattr(torch._C, name)
    assert lib._stream() == (73 if initialised and not missing else 77)
    assert lib._stream(SimpleNamespace(cuda_stream=5)) == 5
