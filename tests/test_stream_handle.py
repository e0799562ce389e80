"""The current stream's handle with a torch that lacks the raw-handle call (host only)."""
import sys
import types

from paper_1803_01756_gb300 import lattice


def fake_torch(raw):
    cuda = types.SimpleNamespace(
        is_initialized=lambda: True, is_available=lambda: True, current_device=lambda: 3,
        current_stream=lambda: types.SimpleNamespace(cuda_stream=1234))
    c = types.SimpleNamespace()
    if raw:
        c._cuda_getCurrentRawStream = lambda device: 5000 + device
    return types.SimpleNamespace(cuda=cuda, _C=c)


def test_falls_back_to_the_stream_object(monkeypatch):
    monkeypatch.setitem(sys.modules, "torch", fake_torch(raw=False))
    assert lattice._stream_ptr(None) == 1234


def test_raw_handle_of_the_current_device(monkeypatch):
    monkeypatch.setitem(sys.modules, "torch", fake_torch(raw=True))
    assert lattice._stream_ptr(None) == 5003
