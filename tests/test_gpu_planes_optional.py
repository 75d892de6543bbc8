"""Batches and servers whose device memory does not hold the tensor-core planes.

The planes are the engine's option there: an image without them is searched in
the plain form.  An allocator with a limit that the plain form's buffers meet
must do for create, and the results stay the oracle's; one that ends before
them gives INPAINT_ERR_NOMEM and leaves nothing allocated.
"""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1403_4238_gb300 import synth

pytestmark = pytest.mark.gpu

NOMEM = -2


class LimitedAllocator:
    """dev_alloc/dev_free over PyTorch's allocator, at most `limit` live bytes and `calls` allocations."""

    def __init__(self, torch):
        from paper_1403_4238_gb300 import _lib
        dev = torch.cuda.current_device()
        self.live, self.peak, self.limit, self.count, self.calls = {}, 0, 1 << 60, 0, 1 << 30

        def alloc(nbytes, stream, user):
            self.count += 1
            now = sum(self.live.values()) + int(nbytes)
            if now > self.limit or self.count > self.calls:
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), dev, int(stream or 0))
            self.live[int(p)] = int(nbytes)
            self.peak = max(self.peak, now)
            return p

        def free(ptr, nbytes, stream, user):
            assert self.live.pop(int(ptr)) == int(nbytes)
            torch.cuda.caching_allocator_delete(int(ptr))

        self.hooks = _lib.ALLOC_FN(alloc), _lib.FREE_FN(free)


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.fixture(scope="module")
def cases():
    out = []
    for k, (W, H, r) in enumerate([(400, 240, 4), (300, 260, 6), (500, 200, 5), (256, 256, 8)]):
        m = np.zeros((H, W), np.uint8)
        m[H // 3:H // 3 + 24, W // 2:W // 2 + 30] = 1
        rgb = synth.image(W, H, 6, 30.0, 40 + k)
        out.append((rgb, m, r, oracle.run(rgb, m, r)))
    return out


def setup(lib, fa, cases):
    from paper_1403_4238_gb300 import _lib
    opt = _lib.Options()
    lib.inpaint_options_default(ctypes.byref(opt))
    opt.dev_alloc, opt.dev_free = fa.hooks
    ims = [_lib.Image(rgb.ctypes.data, m.shape[1], m.shape[0], 3 * m.shape[1], m.ctypes.data, m.shape[1], r)
           for rgb, m, r, _ in cases]
    return opt, (_lib.Image * len(ims))(*ims)


def check_batch(lib, b, cases):
    assert lib.inpaint_batch_run_ctx(b, 0, None) == 0
    for i, (rgb, m, r, ref) in enumerate(cases):
        out = np.zeros_like(rgb)
        it, ev = ctypes.c_int(), ctypes.c_uint64()
        assert lib.inpaint_batch_result(b, i, out.ctypes.data, 3 * m.shape[1], ctypes.byref(it), ctypes.byref(ev)) == 0
        assert it.value == ref.iters and ev.value == ref.evals and np.array_equal(out, ref.rgb), i


def test_batch_without_room_for_planes(torch, cases):
    from paper_1403_4238_gb300 import _lib
    lib, fa = _lib.load(), LimitedAllocator(torch)
    cases = cases * 5
    opt, ims = setup(lib, fa, cases)
    b = ctypes.c_void_p()
    assert lib.inpaint_batch_create(ims, len(ims), ctypes.byref(opt), ctypes.byref(b)) == 0
    calls, full = fa.count, fa.peak
    check_batch(lib, b, cases)
    lib.inpaint_batch_destroy(b)
    # everything but the planes is 42 to 43 bytes a pixel, and the planes are more than 10
    plain = sum(43 * m.size for _, m, _, _ in cases) + (2 << 20)
    assert plain < full
    for limit in (full - 1, plain):
        fa.limit = limit
        assert lib.inpaint_batch_create(ims, len(ims), ctypes.byref(opt), ctypes.byref(b)) == 0, limit
        check_batch(lib, b, cases)
        lib.inpaint_batch_destroy(b)
        assert not fa.live
    fa.limit = plain // 2
    assert lib.inpaint_batch_create(ims, len(ims), ctypes.byref(opt), ctypes.byref(b)) == NOMEM and not b.value
    assert not fa.live
    fa.limit = 1 << 60
    for k in (0, 1, 7, calls // 2, calls - 1):  # no allocation after the k-th
        fa.count, fa.calls = 0, k
        rc = lib.inpaint_batch_create(ims, len(ims), ctypes.byref(opt), ctypes.byref(b))
        assert rc == NOMEM and not b.value and not fa.live, k


def test_server_without_room_for_planes(torch, cases):
    from paper_1403_4238_gb300 import _lib
    lib, fa = _lib.load(), LimitedAllocator(torch)
    rgb, m, r, ref = cases[0]
    opt, ims = setup(lib, fa, cases)
    fa.limit = 43 * m.size + (256 << 10)
    s, rid, info = ctypes.c_void_p(), ctypes.c_uint64(), _lib.RequestInfo()
    assert lib.inpaint_server_create(1 << 30, 4, 0, ctypes.byref(opt), ctypes.byref(s)) == 0
    try:
        assert lib.inpaint_server_submit(s, ctypes.byref(ims[0]), ctypes.byref(rid)) == 0
        assert lib.inpaint_server_wait_idle(s, 60.0) == 0
        out = np.zeros_like(rgb)
        assert lib.inpaint_server_poll(s, rid, out.ctypes.data, 3 * m.shape[1], ctypes.byref(info)) == 0
        assert info.status == 0 and info.iterations == ref.iters and np.array_equal(out, ref.rgb)
    finally:
        lib.inpaint_server_destroy(s)
    assert not fa.live
