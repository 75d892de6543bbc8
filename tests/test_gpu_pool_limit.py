"""Device memory running out without allocator hooks, in a stream-ordered pool
of bounded size: the call that asked for too much reports it, and no later one
does.

The process's pool is replaced by one that holds 64 MB at most for the length
of a test, so cudaMallocAsync fails as on a full device.
"""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1403_4238_gb300 import synth

pytestmark = pytest.mark.gpu


class PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


class SmallPool:
    def __init__(self, torch, bytes_max):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.cu.cuMemAllocFromPoolAsync.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t, ctypes.c_void_p,
                                                    ctypes.c_void_p]
        torch.cuda.synchronize()
        dev = torch.cuda.current_device()
        self.default, self.pool, self.held = ctypes.c_void_p(), ctypes.c_void_p(), []
        props = PoolProps(1, 0, 1, dev, None, bytes_max, 0)  # pinned (device) memory on this device
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.default), dev) == 0
        assert self.cu.cuMemPoolCreate(ctypes.byref(self.pool), ctypes.byref(props)) == 0
        assert self.cu.cuDeviceSetMemPool(dev, self.pool) == 0
        self.dev, self.torch = dev, torch

    def fill(self):
        """Takes what is left of the pool, down to the smallest block."""
        n = 64 << 20
        while n >= 256:
            p = ctypes.c_void_p()
            if self.cu.cuMemAllocFromPoolAsync(ctypes.byref(p), n, self.pool, None) == 0:
                self.held.append(p)
            else:
                n //= 2
        self.torch.cuda.synchronize()

    def free(self):
        for p in self.held:
            assert self.cu.cuMemFreeAsync(p, None) == 0
        self.held = []
        self.torch.cuda.synchronize()

    def close(self):
        self.free()
        assert self.cu.cuDeviceSetMemPool(self.dev, self.default) == 0
        assert self.cu.cuMemPoolDestroy(self.pool) == 0


@pytest.fixture
def pool():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.zeros(1, device="cuda")
    p = SmallPool(torch, 64 << 20)
    yield p
    p.close()


def test_create_after_one_that_did_not_fit(pool):
    from paper_1403_4238_gb300 import _lib, api
    big = synth.tiny(2000, 1500, 3, hole=(700, 600, 90, 80), r=4)  # more than 64 MB of state
    case = synth.small_rect(seed=61)
    ora = oracle.run(case.rgb, case.mask, case.r)
    with pytest.raises(_lib.InpaintError) as e:
        api.Inpainter(big.rgb, big.mask, big.r, torch_memory=False)
    assert e.value.code == _lib.STATUS["ERR_NOMEM"]
    with api.Inpainter(case.rgb, case.mask, case.r, torch_memory=False) as ip:
        assert ip.run()[1] == ora.iters and np.array_equal(ip.result(), ora.rgb)


def test_partial_overlap_goes_on_in_the_graph_loop(pool):
    from paper_1403_4238_gb300 import api
    case = synth.small_rect(seed=61)
    ora = oracle.run(case.rgb, case.mask, case.r, overlap=True)
    with api.Inpainter(case.rgb, case.mask, case.r, torch_memory=False, overlap=True) as ip:
        pool.fill()  # nothing left for the engine's buffers
        assert ip.run()[1] == ora.iters and np.array_equal(ip.result(), ora.rgb)
        pool.free()
