"""Calls without host outputs recorded into a CUDA graph: a replay splits the
tour that was recorded, whatever the context has split in between."""
import numpy as np
import pytest

import oracle
from synth import make_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv():
    from paper_2511_18022_gb300 import build
    build.build()
    import paper_2511_18022_gb300 as m
    return m


# the automatic choice on both sides of its lines, every kernel by request (rings of
# 8 set scenarios aside, whose pass reads the table too), tours around the parts in
# which a recorded table travels
@pytest.mark.parametrize("n,S,config", [
    (100, 37, {}), (100, 1000, {}), (300, 100, {}), (100, 9000, {}), (40, 300, {}),
    (100, 700, dict(kernel=1, threads=64, spt=1, ring=8)), (100, 700, dict(kernel=1, threads=128, spt=2, ring=16)),
    (200, 60, dict(kernel=3)), (2040, 60, {}), (2041, 60, {}), (4080, 40, {}), (4081, 40, {}), (8191, 20, {})])
@pytest.mark.parametrize("mode", ["global", "relaxed"])
def test_replay_after_other_calls(cv, n, S, config, mode):
    Q = 70
    rec, other = (make_instance(n, 1, 10, seed=s, Q=Q) for s in (1, 2))
    xy = rec.coords[rec.tour]                                # deques of many entries
    rec.tour = rec.tour[np.lexsort((xy[:, 0], xy[:, 1] * 3 // (xy[:, 1].max() + 1)))].copy()
    D = np.random.default_rng(n).integers(1, 11, (n, S)).astype(np.int16)
    want = oracle.split_costs(rec.tour, rec.dist, D, Q, n, nthreads=8)[0]
    other_want = oracle.split_costs(other.tour, other.dist, D, Q, n, nthreads=8)[0]
    sp, s = cv.Splitter(0), torch.cuda.Stream()
    sp.configure(**config)
    dev, out, other_out = torch.from_numpy(D).cuda(), torch.empty(S, dtype=torch.int32, device="cuda"), \
        torch.empty(S, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(s):                               # allocates; a waiting call leaves nothing behind that
        sp.split(rec.tour, rec.dist, dev, Q, host_outputs=mode == "global")   # a strict capture would refuse
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode=mode):
        sp.split(rec.tour, rec.dist, dev, Q, out_cost=out, host_outputs=False)
    for wait in (True, False):
        with torch.cuda.stream(s):
            sp.split(other.tour, other.dist, dev, Q, out_cost=other_out, host_outputs=wait)
            out.fill_(-1)
            g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
        assert np.array_equal(other_out.cpu().numpy(), other_want)
    sp.check_inputs()
    sp.close()
