"""max_iters where the caller's stream has work pending.

The limit of a run must reach the device as it was given, also when nothing of
the call has run before the host is through with it: each loop runs two
iterations behind a long kernel on its stream, then one step, then the rest;
the records against the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_1403_4238_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("r,loop,form,overlap", [
    (12, "auto", "plain", False), (4, "graph", "plain", False), (4, "graph", "tc", False),
    (4, "graph", "plain", True), (4, "auto", "plain", True), (4, "engine", "plain", False),
])
def test_limit_behind_pending_work(torch, r, loop, form, overlap):
    from paper_1403_4238_gb300 import api
    case = synth.tiny(130, 110, 5, hole=(40, 30, 30, 34), r=r)
    ora = oracle.run(case.rgb, case.mask, r, overlap=overlap)
    assert ora.iters > 4
    stream = torch.cuda.Stream()
    with api.Inpainter(case.rgb, case.mask, r, loop=loop, form=form, overlap=overlap, stream=stream) as ip:
        ip.run(max_iters=1)  # the graph and the engine's buffers exist
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)  # about 50 ms
        rc, n, tr = ip.run(max_iters=2)
        assert rc == 0 and n == 2
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)
        t = ip.step()
        assert t["iter"] == 3 and (t["qx"], t["qy"]) == (ora.trace[3]["qx"], ora.trace[3]["qy"])
        rc, n, tr = ip.run()
        assert rc == 0 and n == ora.iters - 4
        assert np.array_equal(ip.result(), ora.rgb)
