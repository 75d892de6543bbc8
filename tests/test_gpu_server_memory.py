"""The server's estimate of a request's device memory against what it allocates.

Every device allocation of a server goes through the hooks of its options, so
the bytes that are live can be counted.  While a request runs, hbm_used (the
estimate that admission is decided by) must not lie below them, whatever its
search rectangle, and not more than a third and a megabyte above, as a request
waits for the budget that its estimate needs.
"""
import ctypes
import time

import numpy as np
import pytest

from paper_1403_4238_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("W,H,r,box,alpha", [
    (500, 3000, 4, (100, 2900, 70, 70), 0.2),   # a narrow rectangle far down a tall image
    (1600, 300, 6, (1400, 100, 80, 60), 0.5),   # one far to the right
    (700, 500, 8, (300, 200, 60, 60), -1.0),    # the whole image
    (300, 900, 2, (60, 700, 180, 40), 0.0),     # the object's own box
])
def test_estimate_covers_what_is_allocated(torch, W, H, r, box, alpha):
    from paper_1403_4238_gb300 import _lib
    lib = _lib.load()
    dev = torch.cuda.current_device()
    live, peak = {}, [0]

    def alloc(nbytes, stream, user):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), dev, int(stream or 0))
        live[int(p)] = int(nbytes)
        peak[0] = max(peak[0], sum(live.values()))
        return p

    def free(ptr, nbytes, stream, user):
        live.pop(int(ptr))
        torch.cuda.caching_allocator_delete(int(ptr))

    hooks = _lib.ALLOC_FN(alloc), _lib.FREE_FN(free)
    opt = _lib.Options()
    lib.inpaint_options_default(ctypes.byref(opt))
    opt.search_alpha, opt.dev_alloc, opt.dev_free = alpha, *hooks
    x, y, w, h = box
    rgb, m = synth.image(W, H, 6, 30.0, 3), np.zeros((H, W), np.uint8)
    m[y: y + h, x: x + w] = 1
    s, rid, st = ctypes.c_void_p(), ctypes.c_uint64(), _lib.ServerStats()
    assert lib.inpaint_server_create(1 << 30, 4, 1, ctypes.byref(opt), ctypes.byref(s)) == 0
    try:
        im = _lib.Image(rgb.ctypes.data, W, H, 3 * W, m.ctypes.data, W, r)
        assert lib.inpaint_server_submit(s, ctypes.byref(im), ctypes.byref(rid)) == 0
        used, end = 0, time.time() + 60
        while not (st.completed or st.failed) and time.time() < end:
            assert lib.inpaint_server_stats_get(s, ctypes.byref(st)) == 0
            used = max(used, st.hbm_used)
        assert used >= peak[0] > 0, (used, peak[0])
        assert used <= peak[0] * 4 / 3 + (1 << 20), (used, peak[0])
    finally:
        lib.inpaint_server_destroy(s)
    assert not live
