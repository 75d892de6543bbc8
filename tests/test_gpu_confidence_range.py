"""Imported confidences at the end of the range: infinite ones, and finite ones
whose sum overflows.

C(p) is the ordered FP64 sum of the patch's confidences over its area, with
the infinities that IEEE arithmetic gives; targets, records and confidences
against the oracle, bit for bit, in both loops.  (Images and steps whose front
holds no NaN: an infinite confidence times a data term of zero has no defined
place in the order of priorities.)
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_4238_gb300 import api as _api
    return _api


def state(r, seed, big):
    rng = np.random.default_rng(seed)
    W, H = 8 * r + 24, 7 * r + 22
    rgb = rng.integers(0, 256, (H, W, 3), dtype=np.uint8)
    om = np.zeros((H, W), np.uint8)
    om[H // 2 - r - 2:H // 2 + r + 3, W // 2 - r - 2:W // 2 + r + 3] = 1
    conf = np.where(om != 0, 0.0, rng.uniform(0.2, 1.0, (H, W)))
    conf[H // 2 - r - 3, W // 2] = big
    return rgb, om, conf


@pytest.mark.parametrize("loop", ["engine", "graph"])
@pytest.mark.parametrize("r,seed,big,iters", [
    (2, 0, np.inf, 2), (4, 0, np.inf, 2), (6, 0, np.inf, 2), (8, 0, np.inf, 2),
    (4, 5, 1.7e308, 4), (6, 1, 1.7e308, 4), (8, 0, 1.7e308, 4),
])
def test_large_confidences(api, r, seed, big, iters, loop):
    st = state(r, seed, big)
    ref = oracle.run_from_state(*st, r, max_iters=iters)
    assert ref.iters == iters and np.isinf(ref.trace["confidence"]).any() and not np.isnan(ref.trace["priority"]).any()
    with api.Inpainter(st[0], st[1], r, loop=loop) as ip:
        ip.import_state(*st)
        rc, n, tr = ip.run(max_iters=iters, trace=True)
        assert n == iters
        for f in ("px", "py", "qx", "qy", "ssd"):
            assert np.array_equal(tr[f], ref.trace[f]), f
        for f in ("priority", "confidence"):
            assert np.array_equal(tr[f].view(np.uint64), ref.trace[f].view(np.uint64)), f
        rgb, om, conf = ip.export_state()
        assert np.array_equal(rgb[om == 0], ref.rgb[om == 0]) and np.array_equal(om, ref.mask)
        assert np.array_equal(conf.view(np.uint64), ref.conf.view(np.uint64))
