"""The warp pass over long lists in calls that only enqueue: a warp's share of
the list, by one scenario at a time or, where demands above Q are found, by its
lanes. Against the oracle, bit for bit, with lists of both kinds and mixed."""
import time

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

S = 230_000                                  # rings of 16, also on devices of 152 SMs


@pytest.fixture(scope="module")
def cv():
    from paper_2511_18022_gb300 import build
    build.build()
    import paper_2511_18022_gb300 as m
    return m


def growing(n):
    """Customers ever farther from the depot: every candidate stays in the deque."""
    pts = np.vstack([[0.0, 0.0], np.stack([1000 + 10.0 * np.arange(n), np.full(n, 200.0)], 1)])
    dist = np.rint(np.hypot(*(pts[:, None] - pts[None]).transpose(2, 0, 1))).astype(np.int32)
    return np.arange(1, n + 1, dtype=np.int32), dist


# shares of 0 to 47 scenarios a warp, listed for a demand above Q, a long deque or
# a window beyond the walk's registers
@pytest.mark.parametrize("n", [33, 90])
@pytest.mark.parametrize("bad,long", [(0.0, 0.0), (0.1, 0.0), (0.127, 0.0), (0.3, 0.0), (1.0, 0.0), (0.0, 0.6), (0.4, 0.4),
                                      (0.02, 1.0)])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_costs(cv, n, bad, long, dtype):
    Q = 900
    tour, dist = growing(n)
    rng = np.random.default_rng([n, int(100 * bad), int(100 * long)])
    D = rng.integers(90, 120, (n, S)).astype(dtype)
    D[:, rng.random(S) < long] //= 10                        # windows of the whole tour
    cols = np.flatnonzero(rng.random(S) < bad)
    D[rng.integers(0, n, len(cols)), cols] = Q + 1
    want, ws, wi, _ = oracle.split_costs(tour, dist, D, Q, n, nthreads=8)
    sp = cv.Splitter(0)
    dev, out = torch.from_numpy(D).cuda(), torch.full((S,), -5, dtype=torch.int32, device="cuda")
    for _ in range(2):
        sp.split(tour, dist, dev, Q, n, out_cost=out, host_outputs=False)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
    sp.check_inputs()
    r = sp.split(tour, dist, dev, Q, n)                      # the totals, by the waiting call's passes
    assert (r.sum, r.infeasible) == (ws, wi)
    dev[n - 1, S - 3] = -1
    dev[0, S - 3] = Q + 1                                    # beside a demand above Q
    sp.split(tour, dist, dev, Q, n, out_cost=out, host_outputs=False)
    with pytest.raises(cv.CvrpsdError):
        sp.check_inputs()
    sp.close()


def test_many_infeasible_scenarios_are_settled_in_passing(cv):
    """A quarter of the scenarios infeasible: a call that enqueues the warp pass
    takes no longer than one that waits and walks the list by threads (1.26 and
    1.40 ms); with one warp for each it took 3.4."""
    n, many, Q = 1000, 500_000, 120
    rng = np.random.default_rng(1)
    xy = rng.integers(0, 1001, (n + 1, 2)).astype(np.float64)
    dist = np.rint(np.hypot(*(xy[:, None] - xy[None]).transpose(2, 0, 1))).astype(np.int32)
    tour = (rng.permutation(n) + 1).astype(np.int32)
    D = torch.randint(1, 31, (n, many), dtype=torch.int16, device="cuda")
    cols = torch.randperm(many, device="cuda")[: many // 4]
    D[torch.randint(0, n, (len(cols),), device="cuda"), cols] = Q + 1
    sp, out, best = cv.Splitter(0), torch.empty(many, dtype=torch.int32, device="cuda"), {}
    for wait in (True, False) * 4:
        torch.cuda.synchronize()
        t = time.perf_counter()
        sp.split(tour, dist, D, Q, n, out_cost=out, host_outputs=wait)
        torch.cuda.synchronize()
        best[wait] = min(best.get(wait, 1.0), time.perf_counter() - t)
    assert int((out == 2**31 - 1).sum()) == many // 4
    assert best[False] < 1.5 * best[True]
    sp.close()
