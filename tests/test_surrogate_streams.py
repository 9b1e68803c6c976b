"""Which workspace a surrogate call gets (host only; streams are stand-ins, memory is the
host's): calls on two streams may run at the same time and must not share one, calls on one
stream share one that grows, and a buffer that a capture has seen is not given back.
"""
import contextlib
import types

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture()
def net(monkeypatch):
    from paper_2106_08040_gb300 import build
    build.build()
    from paper_2106_08040_gb300 import surrogate
    state = types.SimpleNamespace(capturing=False, current=types.SimpleNamespace(cuda_stream=0))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: state.current)
    monkeypatch.setattr(torch.cuda, "stream", lambda s: contextlib.nullcontext())
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: state.capturing)
    s = surrogate.Surrogate.__new__(surrogate.Surrogate)
    s.device = torch.device("cpu")
    s._ws, s._captured = {}, {}
    return s, state


def stream(handle):
    return types.SimpleNamespace(cuda_stream=handle)


def test_streams_have_their_own(net):
    s, state = net
    one, two = stream(11), stream(12)
    a, b = s.workspace(300, 0, one), s.workspace(300, 0, two)
    assert a.data_ptr() != b.data_ptr()
    state.current = two
    assert s.workspace(300, 0).data_ptr() == b.data_ptr() and s.workspace(300, 0, one).data_ptr() == a.data_ptr()


def test_one_stream_keeps_one_buffer(net):
    s, _ = net
    for q in (7, 4096, 257, 1, 4095, 100):
        for training in (0, 2, 1) if q % 8 == 0 else (0, 2):
            from paper_2106_08040_gb300 import _lib
            assert s.workspace(q, training, stream(5)).numel() == _lib.lib().fp_surrogate_workspace_bytes(q, training)
    assert [w.tensor.numel() for w in s._ws.values()] == [_lib.lib().fp_surrogate_workspace_bytes(4096, 1)]


def test_a_captured_buffer_is_kept(net):
    s, state = net
    state.capturing = True
    a = s.workspace(64, 0, stream(5))
    state.capturing = False
    b = s.workspace(4096, 0, stream(5))
    assert b.data_ptr() != a.data_ptr()
    assert [w.data_ptr() for w in s._captured.values()] == [a.data_ptr()]


def test_a_refused_size_is_an_error(net):
    s, _ = net
    with pytest.raises(RuntimeError, match="q=0"):
        s.workspace(0, 0, stream(5))
