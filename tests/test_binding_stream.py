"""The stream that a call without one runs on is torch's current stream, with
torch's raw-handle function and, in a torch that lacks it, without."""
import sys
import types

import pytest

from paper_2606_26472_gb300 import epikv as E


class _Stream:
    cuda_stream = 77


@pytest.mark.parametrize("private", [("_cuda_getCurrentRawStream", "_cuda_getDevice"), ("_cuda_getCurrentRawStream",),
                                     ("_cuda_getDevice",), ()])
def test_current_stream_with_and_without_the_raw_function(monkeypatch, private):
    calls = []
    has = {"_cuda_getCurrentRawStream": lambda device: 1000 + device, "_cuda_getDevice": lambda: 3}
    torch = types.SimpleNamespace(
        _C=types.SimpleNamespace(**{n: has[n] for n in private}),
        cuda=types.SimpleNamespace(init=lambda: calls.append("init"), current_stream=lambda: _Stream))
    monkeypatch.setitem(sys.modules, "torch", torch)
    monkeypatch.setattr(E, "_current_stream", None)
    for _ in range(2):
        assert E._stream(None) == (1003 if len(private) == 2 else 77)
    assert calls == ["init"]   # CUDA is initialised first, once
    assert E._stream(5) == 5 and E._stream(_Stream) == 77
