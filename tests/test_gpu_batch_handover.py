"""Two images in turn on one team: nothing of the first is left to be written
when the second one begins.

What a leader writes after its last round of an image (tile maxima, record,
next target) counts when the image is resumed, so runs of a few iterations
over more images than SMs, of mixed sizes and radii and of both forms, are
resumed until every image is done; iterations, evaluations and pixels of all
of them against the oracle, tolerance 0.
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


@pytest.mark.parametrize("max_iters", [1, 5, 0])
def test_images_in_turn_on_one_cta(api, max_iters):
    import torch

    sms = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
    rng = np.random.default_rng(77)
    kinds = []
    for k in range(12):
        r = 1 + k % 8
        W, H = int(rng.integers(6 * r + 24, 150)), int(rng.integers(6 * r + 20, 110))
        m = synth.ellipse_mask(W, H, 2, 0.02, 0.04, 900 + k)
        m[H // 2, W // 8:W - W // 8] = 1  # tiles of several windows
        rgb = synth.image(W, H, 6, 30.0, 800 + k)
        kinds.append((rgb, m, r, oracle.run(rgb, m, r)))
    n = 3 * sms + 5  # three or four images a CTA
    order = [int(k) for k in rng.integers(0, len(kinds), n)]
    with api.Batch([kinds[k][:3] for k in order]) as b:
        plan = b.plan()
        assert plan["teams"] == plan["grid"] and max(plan["team_size"]) == 1
        most = max(kinds[k][3].iters for k in set(order))
        runs = -(-most // max_iters) if max_iters else 1
        for _ in range(runs):
            assert all(x in (0, 1) for x in b.run(max_iters))
        for i, k in enumerate(order):
            out, iters, evals = b.result(i)
            ref = kinds[k][3]
            assert ref.status == 0 and iters == ref.iters and evals == ref.evals, (i, k)
            assert np.array_equal(out, ref.rgb), (i, k)
