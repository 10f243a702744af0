"""The binding's scratch buffers: one per host thread and stream, so that calls that may overlap share none; a bounded number of
them; none kept from a capture, whose memory belongs to the graph.  (Handles and devices are made up: no GPU.)"""
import threading

import pytest

from paper_2106_06998_b200 import binding as xb


@pytest.fixture
def current(monkeypatch):
    state = dict(stream=101, capturing=False)
    monkeypatch.setattr(xb, "_stream", lambda: state["stream"])
    monkeypatch.setattr(xb, "_capturing", lambda: state["capturing"], raising=False)
    return state


def _on_stream(current, handle, nbytes=1000):
    current["stream"] = handle
    return xb.workspace(nbytes, "cpu")


def test_streams_share_no_buffer_and_one_stream_keeps_its_own(current):
    a, b = _on_stream(current, 101), _on_stream(current, 102)
    assert a.data_ptr() != b.data_ptr()
    assert _on_stream(current, 101).data_ptr() == a.data_ptr() and _on_stream(current, 102).data_ptr() == b.data_ptr()
    assert _on_stream(current, 101, 5000).numel() >= 5000 and _on_stream(current, 102).data_ptr() == b.data_ptr()


def test_threads_on_one_stream_share_no_buffer(current):
    mine, theirs = _on_stream(current, 103), []
    t = threading.Thread(target=lambda: theirs.append(xb.workspace(1000, "cpu")))
    t.start()
    t.join()
    assert theirs[0].data_ptr() != mine.data_ptr()


def test_buffers_of_streams_no_longer_used_are_given_back(current):
    import weakref
    refs = []
    for h in range(200, 264):
        refs.append(weakref.ref(_on_stream(current, h)))
    alive = sum(r() is not None for r in refs)
    assert alive <= 8 and refs[-1]() is not None


def test_a_capture_keeps_nothing(current):
    kept = _on_stream(current, 104)
    current["capturing"] = True
    a, b = xb.workspace(1000, "cpu"), xb.workspace(1000, "cpu")
    assert len({kept.data_ptr(), a.data_ptr(), b.data_ptr()}) == 3
    current["capturing"] = False
    assert xb.workspace(1000, "cpu").data_ptr() == kept.data_ptr()
