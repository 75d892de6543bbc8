"""Result arrays faulted in ahead: each is handed out once, keeps its shape,
and none is kept for a request that is gone or after the wait ended."""
import threading
import time

import pytest

from paper_1403_4238_gb300.api import _ResultMemory


def settle(before):
    end = time.time() + 10.0
    while threading.active_count() > before and time.time() < end:
        time.sleep(0.01)


@pytest.mark.parametrize("h,n", [(700, 5), (3, 2)])  # above and below the size that starts a thread
def test_each_array_once(h, n):
    m, before = _ResultMemory(), threading.active_count()
    shapes = {i: (h, 1000 + i, 3) for i in range(n)}
    m.fill(shapes, lambda i: i != 1)
    settle(before)
    m.stop()
    assert 1 not in m._ready and len(m._ready) == (n - 1 if h == 700 else 0)
    got = [m.take(i, s) for i, s in shapes.items()] + [m.take(0, shapes[0])]
    assert [a.shape for a in got] == list(shapes.values()) + [shapes[0]]
    assert len({a.ctypes.data for a in got}) == n + 1 and not any(a.any() for a in got)
    m.put_back(7, got[0])
    assert m.take(7, shapes[0]) is got[0] and not m._ready


def test_nothing_after_stop():
    m, gate, before = _ResultMemory(), threading.Event(), threading.active_count()
    m.fill({i: (700, 1000, 3) for i in range(5)}, lambda i: gate.set() or True)
    assert gate.wait(10.0)
    m.stop()
    have = set(m._ready) | {0}
    settle(before)
    assert len(m._ready) <= len(have) + 1
