"""The resident plain search at the edges of its split into units.

A unit is 32 candidate rows x 4 or 16 candidate columns; the units go to the
searching CTAs in equal contiguous ranges (151 of them for one image on 152
SMs).  Unit counts around that number and its double (CTAs without work, with
one unit, ranges across a band), and around 12 units of 16 columns per CTA,
where the unit grows from 4 columns to 16; ragged last columns and bands.
The first iterations against the oracle, tolerance 0.
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


@pytest.mark.parametrize("r,cols,rows,iters", [
    (1, 4, 32, 8), (4, 4 * 150, 32, 8), (4, 4 * 151, 32, 8), (3, 4 * 151 + 1, 31, 8), (6, 4 * 151 - 3, 33, 8),
    (8, 4 * 50 + 2, 97, 8), (2, 16 * 226, 256, 4), (4, 16 * 227 - 5, 256, 4), (6, 16 * 228, 250, 3),
])
def test_unit_edges(api, r, cols, rows, iters):
    W, H = cols + 2 * r, rows + 2 * r
    rgb = synth.image(W, H, 9, 25.0, cols + rows)
    m = np.zeros((H, W), np.uint8)
    m[0:min(3, r), 0:r] = m[H - 2:, W - r:] = 1
    m[H // 2 - 1:H // 2 + 2, W // 2:W // 2 + 2] = 1
    m[H // 3, W // 4] = 1
    if cols <= 4:
        m[:] = 0
        m[H // 2, 0:2] = 1
    ora = oracle.run(rgb, m, r, max_iters=iters)
    with api.Inpainter(rgb, m, r) as ip:
        rc, n, tr = ip.run(iters, trace=True)
        out = ip.result()
    assert rc == ora.status and n == ora.iters
    for f in ("px", "py", "qx", "qy", "ssd", "filled", "remaining", "n_known", "n_cand"):
        assert [t[f] for t in tr] == [t[f] for t in ora.trace], f
    assert (out == ora.rgb).all()
