"""Result arrays faulted in ahead: how much is held, for whom, and until when."""
import threading
import time

import pytest

from paper_1403_4238_gb300.api import _ResultMemory


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
