"""The partial-overlap search in the engine against the graph loop and the oracle.

Every patch radius with candidate columns that start off a 16-byte boundary
(the rectangle begins at the image border), ragged last unit columns and
bands, lanes and rows that are wholly inside the object or outside the image,
objects across bands and on every border, search rectangles of both kinds, and
resumed runs; tolerance 0.
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


@pytest.mark.parametrize("r,W,H,alpha", [
    (1, 61, 35, -1.0), (2, 130, 64, -1.0), (3, 97, 66, 0.4), (4, 203, 97, -1.0), (5, 150, 33, -1.0),
    (6, 259, 70, 0.7), (7, 122, 95, -1.0), (8, 301, 65, -1.0), (8, 17, 40, -1.0),
])
def test_loops_agree(api, r, W, H, alpha):
    rgb = synth.image(W, H, 7, 30.0, 300 + W)
    m = np.zeros((H, W), np.uint8)
    m[H // 2:H // 2 + min(5, H // 8), W // 8:W - W // 8] = 1  # a strip: whole lanes without a source
    m[0:3, W - 4:] = m[H - 2:, 0:3] = 1
    if alpha < 0 and H > 80:
        m[30:36, W // 3:W // 3 + 3] = 1  # across a band of 32 rows
    ora = oracle.run(rgb, m, r, alpha=alpha, overlap=True)
    outs = []
    for loop, cut in (("auto", 0), ("auto", 3), ("graph", 0)):
        with api.Inpainter(rgb, m, r, alpha=alpha, overlap=True, loop=loop) as ip:
            got = []
            while True:
                rc, n, tr = ip.run(cut, trace=True)
                got += list(tr[:n])
                if rc != 0 or n == 0 or ip.info()["remaining"] == 0:
                    break
            outs.append((rc, got, ip.result(), ip.info()["evals"]))
    for rc, got, out, evals in outs:
        assert len(got) == ora.iters
        for f in FIELDS:
            assert [t[f] for t in got] == [t[f] for t in ora.trace], f
        for f in ("priority", "confidence"):
            assert [np.float64(t[f]).view(np.uint64) for t in got] == \
                   [np.float64(t[f]).view(np.uint64) for t in ora.trace], f
        assert (out == ora.rgb).all() and evals == ora.evals


def test_graph_loop_where_the_engine_cannot(api):
    """Engine options that only the engine checks do not stop the variant: the graph loop runs it."""
    rgb, m = synth.image(90, 60, 7, 30.0, 5), np.zeros((60, 90), np.uint8)
    m[20:26, 30:44] = 1
    ora = oracle.run(rgb, m, 3, overlap=True)
    with api.Inpainter(rgb, m, 3, overlap=True, tile_rows=3) as ip:
        rc, n, tr = ip.run(trace=True)
        assert rc == 0 and n == ora.iters and (ip.result() == ora.rgb).all()
