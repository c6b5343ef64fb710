"""The stream argument of the Python calls on the host: the current stream with
and without PyTorch's internal query."""
from types import SimpleNamespace

import pytest

import paper_1002_0916_gb300 as cg


@pytest.mark.parametrize("initialized", [False, True])
@pytest.mark.parametrize("internal", [False, True])
def test_current_stream(monkeypatch, initialized, internal):
    c = SimpleNamespace(_cuda_getDevice=lambda: 3, _cuda_getCurrentRawStream=lambda d: 70 + d)
    torch = SimpleNamespace(
        _C=c if internal else SimpleNamespace(),
        cuda=SimpleNamespace(is_initialized=lambda: initialized,
                             current_stream=lambda: SimpleNamespace(cuda_stream=73)))
    monkeypatch.setattr(cg, "_torch", lambda: torch)
    assert cg._stream_ptr(None) == 73
    assert cg._stream_ptr(SimpleNamespace(cuda_stream=5)) == 5
    assert cg._stream_ptr(9) == 9
