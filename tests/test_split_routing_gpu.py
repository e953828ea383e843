"""Which kernel and launch shape a single-tour call takes, at the sizes where
the choice changes, and what one call leaves for the next: against the oracle,
bit for bit."""
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


def instance(n, Q, kind, seed):
    inst = make_instance(n, 1, 10, seed=seed, Q=Q)
    if kind == "smooth":                                     # in strips: C_i rises along them
        xy = inst.coords[inst.tour]
        inst.tour = inst.tour[np.lexsort((xy[:, 0], xy[:, 1] * 3 // (xy[:, 1].max() + 1)))].copy()
    if kind == "flat":                                       # C_i = 0 everywhere, equal costs
        inst.dist = np.zeros((n + 1, n + 1), np.int32)
        inst.dist[0, 1:] = inst.dist[1:, 0] = 1
    return inst


def demands(n, S, Q, dtype, seed):
    D = np.random.default_rng(seed).integers(0, 20, (n, S)).astype(dtype)
    D[:, 1] = 0
    D[n // 2, 2] = Q + 1
    D[n - 1, S - 1] = 32767
    return D


@pytest.mark.parametrize("dtype", [np.int16, np.int32])
@pytest.mark.parametrize("kind", ["random", "smooth", "flat"])
@pytest.mark.parametrize("more", [0, 1])                     # all scenarios resident with rings of 32, and one more
@pytest.mark.parametrize("L", [None, 9])
def test_rings_of_32_and_16(cv, more, kind, L, dtype):
    n, Q = 45, 160
    S = 64 * 14 * torch.cuda.get_device_properties(0).multi_processor_count + more
    inst = instance(n, Q, kind, 5)
    D = demands(n, S, Q, dtype, 6)
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, L or n, nthreads=8)
    sp = cv.Splitter(0)
    out = torch.empty(S, dtype=torch.int32, device="cuda")
    r = sp.split(inst.tour, inst.dist, torch.from_numpy(D).cuda(), Q, L, out_cost=out)
    assert sp.stats()["ring"] == (32 if dtype == np.int16 and not more else 16)
    assert np.array_equal(out.cpu().numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    sp.close()


@pytest.mark.parametrize("kind", ["random", "smooth", "flat"])
@pytest.mark.parametrize("n,S", [(1, 70), (9, 65), (1023, 70), (1024, 70), (1025, 70), (30, 136_193)])
def test_predecessors(cv, n, S, kind):
    Q = 160
    inst = instance(n, Q, kind, n)
    D = demands(n, S, Q, np.int16, n)
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, n, nthreads=8)
    sp = cv.Splitter(0)
    pred = torch.full((n, S + 3), -9, dtype=torch.int16, device="cuda")
    out = torch.empty(S, dtype=torch.int32, device="cuda")
    r = sp.split_routes(inst.tour, inst.dist, torch.from_numpy(D).cuda(), Q, pred=pred, out_cost=out)
    P = pred.cpu().numpy()
    assert np.array_equal(out.cpu().numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    assert (P[:, S:] == -9).all()
    for s in (0, 1, S // 2, S - 2):
        cost, _, opred = oracle.split_routes(inst.tour, inst.dist, D[:, s], Q, n)
        assert cost is None or np.array_equal(P[:, s], opred[1:]), f"scenario {s}"
    sp.close()


def test_calls_in_a_row(cv):
    """Waiting and enqueueing calls of every kernel in turn, with set-aside and
    negative demands in between, on two streams: totals never carry over."""
    n, Q = 80, 120
    inst = instance(n, Q, "smooth", 3)
    sp, other = cv.Splitter(0), torch.cuda.Stream()
    for k, S in enumerate((50, 700, 9000, 140_000, 9000, 50)):
        D = demands(n, S, Q, np.int16, k)
        want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, n, nthreads=8)
        dev = torch.from_numpy(D).cuda()
        out = torch.empty(S, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(other if k % 2 else torch.cuda.current_stream()):
            sp.split(inst.tour, inst.dist, dev, Q, out_cost=out, host_outputs=False)
            r = sp.split(inst.tour, inst.dist, dev, Q)
            assert (r.sum, r.infeasible) == (ws, wi)
            assert np.array_equal(out.cpu().numpy(), want)
            bad = dev.clone()
            bad[1, 0] = -1
            with pytest.raises(cv.CvrpsdError):
                sp.split(inst.tour, inst.dist, bad, Q)
            with pytest.raises(cv.CvrpsdError):
                sp.check_inputs()
            r = sp.split(inst.tour, inst.dist, dev, Q, out_cost=out)
            assert (r.sum, r.infeasible) == (ws, wi)
            assert np.array_equal(out.cpu().numpy(), want)
        torch.cuda.synchronize()
    sp.close()
