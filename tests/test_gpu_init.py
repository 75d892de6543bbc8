"""Initialisation on the device: counts from Omega's bit rows, the initial
front, its priorities and the first target.

Radii around the word size of a patch row (2 r + 1 = 31, 33, 63, 65 bits),
widths around the words, the count's columns (128) and the priority windows
(4 r + 3), heights around its rows (16) and the level-1 tiles (256), masks on
the image border and in the last partial word.  The debug checks recount every
centre's unknown pixels and evaluate every priority from scratch after each
step; the records against the oracle, tolerance 0.
"""
import numpy as np
import pytest

import oracle
from paper_1403_4238_gb300 import synth

pytestmark = pytest.mark.gpu

FIELDS = ("px", "py", "qx", "qy", "ssd", "filled", "remaining", "n_known", "n_cand")


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_4238_gb300 import api as _api
    return _api


@pytest.mark.parametrize("W,H,r", [
    (97, 16, 1), (128, 33, 2), (129, 47, 4), (127, 49, 7), (257, 40, 8), (300, 261, 8), (160, 80, 15),
    (161, 65, 16), (193, 70, 31), (224, 97, 32), (257, 81, 32),
])
def test_initial_state(api, W, H, r):
    rgb = synth.image(W, H, 6, 30.0, W + r)
    m = np.zeros((H, W), np.uint8)
    m[H // 2, W // 2:W // 2 + 3] = 1
    m[0, 0] = m[H - 1, W - 1] = m[H - 2, W - 1] = 1
    m[0, 31:34] = 1
    m[H // 3:H // 3 + 2, 63:66] = 1
    ora = oracle.run(rgb, m, r, max_iters=3)
    with api.Inpainter(rgb, m, r, debug=1) as ip:
        for i in range(min(3, ora.iters)):
            t = ip.step()
            for f in FIELDS:
                assert t[f] == ora.trace[i][f], (i, f)
            for f in ("priority", "confidence"):
                assert np.float64(t[f]).view(np.uint64) == np.float64(ora.trace[i][f]).view(np.uint64), (i, f)
