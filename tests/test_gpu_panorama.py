"""Images with a side beyond 32767: targets far along it, in every loop and form.

The engine's leader tells the searchers the next target in one word; columns
and rows of every accepted image (2^30 pixels) must fit it.  Objects at both
ends and in the middle, sides next to a power of two; every record and the
pixels against the oracle, tolerance 0.
"""
import numpy as np
import pytest

import oracle
from paper_1403_4238_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_4238_gb300 import api as _api
    return _api


def strip(W, H, seed):
    """A long image with objects along it (the pattern repeats, moved a little each time)."""
    n = max(W, H)
    tile = synth.image(1024, min(W, H), 7, 30.0, seed)
    rgb = np.concatenate([np.roll(tile, 97 * k, axis=1) for k in range(-(-n // 1024))], axis=1)[:, :n].copy()
    m = np.zeros((min(W, H), n), np.uint8)
    for x in (40, n // 2, n - 3000, n - 60):
        m[9:15, x:x + 12] = 1
    if H > W:
        rgb, m = np.ascontiguousarray(rgb.transpose(1, 0, 2)), np.ascontiguousarray(m.T)
    return rgb, m


@pytest.mark.parametrize("W,H,r", [(40001, 25, 2), (32769, 33, 4), (29, 45000, 3)])
def test_long_images(api, W, H, r):
    rgb, m = strip(W, H, W + H)
    ora = oracle.run(rgb, m, r)
    for form, loop in (("plain", "engine"), ("plain", "graph"), ("tc", "engine")):
        with api.Inpainter(rgb, m, r, form=form, loop=loop) as ip:
            rc, n, tr = ip.run(trace=True)
            assert rc == 0 and n == ora.iters, (form, loop)
            for f in ("px", "py", "qx", "qy", "ssd", "n_cand"):
                assert np.array_equal(tr[f], ora.trace[f]), (form, loop, f)
            assert np.array_equal(ip.result(), ora.rgb), (form, loop)
    with api.Batch([(rgb, m, r)] * 3) as b:
        assert b.run() == [0, 0, 0]
        for i in range(3):
            out, iters, evals = b.result(i)
            assert iters == ora.iters and evals == ora.evals and np.array_equal(out, ora.rgb)


def test_long_image_partial_overlap(api):
    rgb, m = strip(36000, 21, 9)
    ora = oracle.run(rgb, m, 2, overlap=True)
    for loop in ("auto", "graph"):
        with api.Inpainter(rgb, m, 2, overlap=True, loop=loop) as ip:
            rc, n, tr = ip.run(trace=True)
            assert rc == 0 and n == ora.iters
            for f in ("px", "py", "qx", "qy", "ssd", "n_cand"):
                assert np.array_equal(tr[f], ora.trace[f]), (loop, f)
            assert np.array_equal(ip.result(), ora.rgb), loop
