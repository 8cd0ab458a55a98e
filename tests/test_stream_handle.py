"""How the binding finds the current stream: through torch's public call first
(which initialises torch's CUDA state), by the handle alone afterwards, and by
the public call where this torch has no such name."""
import types

import pytest

from paper_2603_15447_gb300 import bez


@pytest.mark.parametrize("has_name", [True, False])
def test_current_stream(monkeypatch, has_name):
    calls = []

    def current_stream(device):
        calls.append(device)
        return types.SimpleNamespace(cuda_stream=100 + device)

    private = types.SimpleNamespace(_cuda_getCurrentRawStream=lambda device: 100 + device) if has_name else \
        types.SimpleNamespace()
    fake = types.SimpleNamespace(cuda=types.SimpleNamespace(current_stream=current_stream), _C=private)
    monkeypatch.setattr(bez, "_torch", lambda: fake)
    monkeypatch.setattr(bez, "_raw_stream", None, raising=False)
    assert bez._stream_handle(None, 0) == 100 and calls == [0]
    assert bez._stream_handle(None, 1) == 101 and calls == ([0] if has_name else [0, 1])
    assert bez._stream_handle(7, 0) == 7
    assert bez._stream_handle(types.SimpleNamespace(cuda_stream=9), 0) == 9
