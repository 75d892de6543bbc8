"""Patch radii above 8: the search in chunks of eight target columns and the
priorities of listed front pixels.

Patch widths with every kind of last chunk (1 to 7 columns, 33 and 65: a
further word of known bits), targets cut by each image border, candidate
rectangles with ragged tiles; whole removals against the oracle, tolerance 0.
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


@pytest.mark.parametrize("r,W,H", [(10, 90, 61), (11, 131, 70), (13, 97, 88), (16, 140, 101), (19, 133, 94),
                                   (31, 201, 140), (32, 213, 133)])
def test_whole_removal(api, r, W, H):
    rgb = synth.image(W, H, 8, 35.0, 40 + r)
    m = np.zeros((H, W), np.uint8)
    m[0:5, 3:9] = m[H - 4:, W // 3:W // 3 + 6] = m[H // 2:H // 2 + 3, 0:4] = 1
    m[H // 2 - 3:H // 2 + 4, W - r // 2:] = 1
    ora = oracle.run(rgb, m, r)
    with api.Inpainter(rgb, m, r) as ip:
        rc, n, tr = ip.run(trace=True)
        out, left = ip.result(with_mask=True)
    assert rc == ora.status and n == ora.iters
    for f in ("px", "py", "qx", "qy", "ssd", "filled", "remaining", "n_known", "n_cand"):
        assert [t[f] for t in tr] == [t[f] for t in ora.trace], f
    for f in ("priority", "confidence"):
        assert [np.float64(t[f]).view(np.uint64) for t in tr] == [np.float64(t[f]).view(np.uint64) for t in ora.trace]
    assert (out == ora.rgb).all() and (left == ora.mask).all()


@pytest.mark.parametrize("r,W,H", [(9, 75, 66), (17, 120, 101)])
def test_steps_and_applied_keys(api, r, W, H):
    """The same iterations outside the graph: search and speculative part on two streams, and applied alone."""
    rgb = synth.image(W, H, 8, 35.0, 70 + r)
    m = np.zeros((H, W), np.uint8)
    m[0:4, 5:9] = m[H // 2:H // 2 + 9, W // 2:W // 2 + 5] = m[H - 3:, W - 6:] = 1
    ora = oracle.run(rgb, m, r)
    with api.Inpainter(rgb, m, r, debug=True) as a, api.Inpainter(rgb, m, r, debug=True) as b:
        for i in range(ora.iters):
            t = a.step()
            u = b.apply_key(b.search_rows(0, H))
            for f in ("px", "py", "qx", "qy", "ssd", "priority", "confidence", "filled", "n_cand"):
                assert t[f] == ora.trace[i][f] and u[f] == ora.trace[i][f], (i, f)
        assert a.step() is None
        assert (a.result() == ora.rgb).all() and (b.result() == ora.rgb).all()
