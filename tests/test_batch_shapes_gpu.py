"""The batch kernels on the second walk, both demand types, at the launch shapes
the library picks (64, 128, 512 or 256 threads by the scenarios at hand), over
tours in random order, tours along lines (whose C_i rise) and a mix of both,
with infeasible demands and rings that overflow. Against the oracle, bit for
bit, through both entry points."""
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


def along(inst, every):
    """The instance's customers in order of x, in `every` strips of y."""
    xy = inst.coords[inst.tour]
    strip = (xy[:, 1] * every // (xy[:, 1].max() + 1)).astype(int)
    return inst.tour[np.lexsort((xy[:, 0], strip))].copy()


def demands(rng, n, S, Q, dtype):
    D = rng.integers(0, 12, (n, S)).astype(dtype)
    D[:, 1] = 0                                              # one window as long as the tour
    D[n // 2, 2] = Q + 1                                     # infeasible
    D[0, 3] = 32767 if dtype == np.int16 else 2**31 - 1
    return D


@pytest.mark.parametrize("dtype", [np.int16, np.int32])
@pytest.mark.parametrize("kind", ["random", "smooth", "mixed"])
@pytest.mark.parametrize("T,S,L", [(3, 5000, None), (5, 20_000, 30), (6, 60_000, None), (6, 60_000, 40)])
def test_batches(cv, T, S, L, kind, dtype):
    rng = np.random.default_rng([T, S, len(kind)])
    sp = cv.Splitter(0)
    tours, wants = [], []
    for t in range(T):
        n = [1, 97, 64, 130, 33, 200][t]
        inst = make_instance(n, 1, 10, seed=40 + t, Q=150)
        tour = along(inst, 3) if kind == "smooth" or (kind == "mixed" and t % 2) else inst.tour
        D = demands(rng, n, S, 150, dtype)
        lim = n if L is None else min(L, n)
        wants.append(oracle.split_costs(tour, inst.dist, D, 150, lim, nthreads=8)[:3])
        tours.append(dict(tour=tour, dist=inst.dist, demand=torch.from_numpy(D).cuda(), Q=150, L=lim,
                          out_cost=torch.full((S,), -3, dtype=torch.int32, device="cuda")))
    b = sp.batch(tours, S)
    for _ in range(2):
        b.run()
        res = b.results()
        for t, (want, ws, wi) in enumerate(wants):
            assert np.array_equal(tours[t]["out_cost"].cpu().numpy(), want), f"tour {t}"
            assert (res["sum"][t], res["infeasible"][t]) == (ws, wi) and wi >= 1
    b.close()
    sp.close()


@pytest.mark.parametrize("dtype", [np.int16, np.int32])
@pytest.mark.parametrize("kind", ["random", "smooth", "mixed"])
@pytest.mark.parametrize("T,S,L", [(5, 900, None), (8, 17_000, 25), (16, 26_285, None)])
def test_tours_of_one_instance(cv, T, S, L, kind, dtype):
    n, Q = 145, 159
    rng = np.random.default_rng([T, S, len(kind)])
    inst = make_instance(n, 1, 10, seed=9, Q=Q)
    D = demands(rng, n, S, Q, dtype)
    tours = np.stack([along(inst, 2 + t % 3) if kind == "smooth" or (kind == "mixed" and t % 2)
                      else rng.permutation(n) + 1 for t in range(T)]).astype(np.int32)
    sp = cv.Splitter(0)
    mean = torch.empty(T, dtype=torch.float64, device="cuda")
    tot = torch.empty(T, dtype=torch.int64, device="cuda")
    bad = torch.empty(T, dtype=torch.int64, device="cuda")
    cv.cvrpsd_split_eval_tours(sp.ctx, torch.from_numpy(tours).cuda(), inst.dist, torch.from_numpy(D).cuda(), Q, L,
                               mean=mean, sums=tot, infeasible=bad)
    torch.cuda.synchronize()
    for t in range(T):
        _, ws, wi, _ = oracle.split_costs(tours[t], inst.dist, D, Q, L or n, nthreads=8)
        assert (int(tot[t]), int(bad[t])) == (ws, wi), f"tour {t}"
    sp.close()
