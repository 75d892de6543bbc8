"""The batched form's tensor-core search at the edges of its geometry.

A batch lets the engine choose the search form per image; images whose round
is shorter in the tensor-core form run it with narrow images folded (several
row blocks side by side in one tile), several tiles per CTA, and leaders that
search.  Widths around the fold limits (64 and 128 blocks of 8 candidate
columns), heights that leave a ragged last fold and a ragged last tile, holes
across the fold boundaries and at the image border; every image against the
oracle, tolerance 0.
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


def photo(W, H, r, seed):
    m = np.zeros((H, W), np.uint8)
    g = np.random.Generator(np.random.PCG64(seed))
    # a thin hole down the whole height (every fold boundary) and one in a corner
    x = int(g.integers(2 * r + 2, max(2 * r + 3, W - 3 * r)))
    m[H // 8:H - H // 8, x:x + 2] = 1
    m[0:r, W - r - 1:W] = 1
    return synth.image(W, H, 7, 30.0, seed), m, r


@pytest.mark.parametrize("r", [1, 2, 4, 5, 6, 7, 8])
def test_batch_folded_and_wide_images(api, r):
    n1 = (2 * r + 1 + 14) // 8 - 1  # blocks a fold needs beyond its candidates
    widths = [2 * r + 8 * (64 - n1), 2 * r + 8 * (64 - n1) + 1, 2 * r + 8 * (42 - n1), 2 * r + 8 * (32 - n1) - 3,
              61 + 2 * r, 1024 + 2 * r, 1025 + 2 * r]
    heights = [57 + 2 * r, 64 + 2 * r, 97 + 2 * r, 81 + 2 * r, 130 + 2 * r, 40 + 2 * r, 33 + 2 * r]
    cases = [photo(W, H, r, 100 * r + k) for k, (W, H) in enumerate(zip(widths, heights))]
    want = [oracle.run(*c) for c in cases]
    for copies in (1, 25):  # teams of about 20 CTAs, and single-CTA teams with searching leaders
        with api.Batch(cases * copies) as b:
            st = b.run()
            assert all(x == 0 for x in st), st
            for i in range(len(cases)):
                out, iters, evals = b.result(i + (copies - 1) * len(cases))
                assert iters == want[i].iters and evals == want[i].evals, i
                assert np.array_equal(out, want[i].rgb), i
            b.reset()  # the planes and the validity bits start over
            b.run()
            assert np.array_equal(b.result(0)[0], want[0].rgb)


@pytest.mark.parametrize("W,H,r", [(480, 90, 4), (480, 90, 6), (700, 60, 5), (250, 300, 8)])
def test_single_image_narrow_tiles(api, W, H, r):
    # one image over all CTAs: several narrow tile columns, MMA widths that
    # are not multiples of 32
    rgb, mask, r = photo(W, H, r, W + r)
    ref = oracle.run(rgb, mask, r)
    for loop in ("engine", "graph"):
        with api.Inpainter(rgb, mask, r, form="tc", loop=loop) as ip:
            rc, n, tr = ip.run(trace=True)
            assert rc == 0 and n == ref.iters
            assert np.array_equal(ip.result(), ref.rgb)
            assert np.array_equal(tr["ssd"], ref.trace["ssd"])
