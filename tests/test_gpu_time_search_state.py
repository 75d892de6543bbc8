"""Timing a search in isolation leaves the removal as it was: counts and
evaluations of the iterations that follow are the oracle's, bit for bit."""
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


@pytest.mark.parametrize("overlap,loop", [(True, "auto"), (True, "graph"), (False, "auto")])
@pytest.mark.parametrize("step_first", [False, True])
def test_counts_after_timing(api, overlap, loop, step_first):
    case = synth.small_rect(seed=61)
    ora = oracle.run(case.rgb, case.mask, case.r, overlap=overlap)
    with api.Inpainter(case.rgb, case.mask, case.r, overlap=overlap, loop=loop) as ip:
        k = 0
        if step_first:
            assert ip.step()["n_cand"] == ora.trace[0]["n_cand"]
            k = 1
        _, key, _ = ip.time_search("plain", 3)
        W = case.mask.shape[1]
        assert key == (int(ora.trace[k]["ssd"]) << 32) | (int(ora.trace[k]["qy"]) * W + int(ora.trace[k]["qx"]))
        t = ip.step()
        for f in ("px", "py", "qx", "qy", "ssd", "n_cand", "n_known"):
            assert t[f] == ora.trace[k][f], f
        ip.time_search("plain", 2)
        rc, n, tr = ip.run(trace=True)
        assert n == ora.iters - k - 1 and np.array_equal(tr["n_cand"], ora.trace["n_cand"][k + 1:])
        assert ip.info()["evals"] == ora.evals and np.array_equal(ip.result(), ora.rgb)


@pytest.mark.parametrize("W,H,r,hole", [(130, 96, 4, (0, 0, 20, 16)), (61, 150, 8, (30, 100, 20, 30)), (64, 40, 1, (50, 30, 14, 10))])
def test_tensor_core_timing_of_a_partial_overlap_context(api, W, H, r, hole):
    """The full search's best patch, whose rectangle ends r pixels before the border."""
    case = synth.tiny(W, H, 7, hole=hole, r=r)
    with api.Inpainter(case.rgb, case.mask, r, overlap=True) as ip:
        rgb, om, _ = ip.export_state()
        _, key, _ = ip.time_search("tc", 2)
        t = ip.step()
        ssd, n_cand, _ = oracle.ssd_map(rgb, om, r, int(t["px"]), int(t["py"]))
        flat = np.where(ssd.ravel() == 0xFFFFFFFF, np.uint64(1 << 40), ssd.ravel().astype(np.uint64))
        assert n_cand > 0 and key == (int(flat.min()) << 32) | int(flat.argmin())
        ora = oracle.run(case.rgb, case.mask, r, overlap=True)
        ip.run()
        assert np.array_equal(ip.result(), ora.rgb)
