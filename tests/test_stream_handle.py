"""The binding's current-stream handle, on the CPU: with torch's raw-stream
functions and without them."""
import types

import pytest
import torch

from paper_2607_20940_gb300 import msf


@pytest.mark.parametrize("missing", [None, "_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_handle(monkeypatch, missing):
    monkeypatch.setattr(msf, "_current", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 77 if d == 3 else 0, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    if missing:
        monkeypatch.delattr(torch._C, missing)
    assert msf._stream(None) == 77 and msf._stream(None) == 77
    assert msf._stream(5) == 5 and msf._stream(types.SimpleNamespace(cuda_stream=9)) == 9


def test_without_cuda(monkeypatch):
    """Initialising CUDA fails: so does every call, not only the first."""
    def fail():
        raise RuntimeError("no CUDA")
    monkeypatch.setattr(msf, "_current", None)
    monkeypatch.setattr(torch.cuda, "current_stream", fail)
    for _ in range(2):
        with pytest.raises(RuntimeError):
            msf._stream(None)
