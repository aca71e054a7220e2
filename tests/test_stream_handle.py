"""The stream handle that the binding passes on: the caller's stream, the current stream's raw
handle, and the same through torch's public names where the raw accessors are missing (no GPU)."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

from paper_2606_18587_gb300 import dar  # noqa: E402


def test_given_stream():
    assert dar._stream(SimpleNamespace(cuda_stream=77)) == 77


def test_raw_handle_of_the_current_device(monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 1000 + device, raising=False)
    assert dar._stream() == 1003


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_without_the_raw_accessors(monkeypatch, missing):
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 1, raising=False)
    monkeypatch.delattr(torch._C, missing)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=55))
    assert dar._stream() == 55
