"""Result arrays faulted in ahead: how much is held, for whom, and until when."""
import threading
import time

import pytest

from paper_1403_4238_gb300 import _lib
from paper_1403_4238_gb300.api import Server, _ResultMemory


def settle(before):
    end = time.time() + 10.0
    while threading.active_count() > before and time.time() < end:
        time.sleep(0.01)


@pytest.mark.parametrize("limit,kept", [(30, 4), (31, 5), (7, 0)])
def test_total_is_bounded(monkeypatch, limit, kept):
    monkeypatch.setattr(_ResultMemory, "MAX_BYTES", limit * 10**6, raising=False)
    m, before = _ResultMemory(), threading.active_count()
    shapes = {i: (2000 + i, 1030, 3) for i in range(9)}  # 6.2 MB each
    m.fill(shapes, lambda i: True)
    settle(before)
    assert list(m._ready) == list(range(kept))
    if kept:
        a = m.take(1, shapes[1])  # its place goes to the next one that is missing
        m.MIN_BYTES = 0
        m.fill({k: v for k, v in shapes.items() if k != 1}, lambda i: True)
        settle(before)
        assert sorted(m._ready) == [0, 2, 3, *range(4, kept + 1)] and a.shape == shapes[1]
    m.stop()


class PolledLib:
    """inpaint_server_poll of a fake library; `during` runs inside each call."""

    def __init__(self, codes, during):
        self.codes, self.during = list(codes), during

    def inpaint_server_poll(self, *args):
        self.during()
        return self.codes.pop(0)


def polled_server(codes, during=lambda: None):
    srv = Server.__new__(Server)  # without a device
    srv.lib, srv.s, srv.shapes, srv._memory = PolledLib(codes, during), None, {5: (2000, 1500), 6: (2000, 1500)}, _ResultMemory()
    return srv


def test_none_is_kept_for_a_request_that_was_polled():
    before = threading.active_count()

    def during():  # another thread's wait_idle finishes the array between the look for it and the end of the poll
        srv._memory.fill({5: (2000, 1500, 3)}, lambda k: k in srv.shapes)
        settle(before)

    srv = polled_server([_lib.STATUS["OK"]], during)
    out, _ = srv.poll(5)
    assert out.shape == (2000, 1500, 3) and 5 not in srv.shapes
    assert not srv._memory._ready


def test_pending_polls_keep_only_what_was_faulted_in():
    before = threading.active_count()
    srv = polled_server([_lib.STATUS["PENDING"]] * 3 + [_lib.STATUS["OK"]])
    assert srv.poll(5) is None and not srv._memory._ready
    srv._memory.fill({k: (*v, 3) for k, v in srv.shapes.items()}, lambda k: k in srv.shapes)  # 5 is not left out
    settle(before)
    a = srv._memory._ready[5]
    assert srv.poll(5) is None and srv.poll(5) is None and srv._memory._ready[5] is a
    assert srv.poll(5)[0] is a and list(srv._memory._ready) == [6]


def test_stop_ends_its_own_fill_and_waits_for_it():
    m, before = _ResultMemory(), threading.active_count()
    gate, started = threading.Event(), threading.Event()

    def hold(i):
        started.set()
        gate.wait(10.0)
        return True

    m.fill({i: (4000, 2000, 3) for i in range(40)}, lambda i: True)  # a wait of one thread
    m.stop()
    assert threading.active_count() == before  # not even in the middle of an array
    first = m.fill({i: (1000, 3000, 3) for i in range(3)}, hold)
    assert started.wait(10.0)
    gate.set()
    second = m.fill({i: (1000, 3000, 3) for i in range(10, 13)}, lambda i: True)  # and of another
    m.stop(first)
    settle(before)
    assert {10, 11, 12} <= set(m._ready)  # the other thread's wait had them made all the same
    m.stop(second)
    assert threading.active_count() == before
