"""Scenarios in host memory whose rows straddle the link's 64-byte lines: the
walk that stages whole lines must equal the oracle and the device entry point
bit for bit, at row ends, group ends and blocks that are partly filled."""
import numpy as np
import pytest

import oracle
from synth import KIND_NORMAL, demand_matrix, make_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_18022_gb300 import build
    build.build()
    import paper_2511_18022_gb300 as m
    return m


# (n, S, pitch, elements before the matrix): full and partly filled last blocks,
# a last block of one scenario, odd pitches, matrices that start on 16, 64 and 2
# bytes (the last is read directly), tours around a group of 8 and the ring of 16.
CASES = [(1, 24577, 24577, 0), (7, 24576, 24577, 8), (8, 24633, 24640, 8), (9, 25089, 25097, 32),
         (25, 24577, 24578, 0), (33, 24600, 24601, 1), (40, 30001, 30001, 16), (130, 24575, 24575, 0)]


@pytest.mark.parametrize("dtype", [np.int16, np.int32])
@pytest.mark.parametrize("n,S,ld,off", CASES)
@pytest.mark.parametrize("cap", [False, True])
def test_staged_rows(cv, n, S, ld, off, dtype, cap):
    inst = make_instance(n, 5, 30, 5, Q=90, L=min(4, n) if cap else n)
    D = demand_matrix(inst.mu, inst.region, KIND_NORMAL, 3, S, dtype=dtype)
    D[n // 2, S - 1] = 91                                    # infeasible
    D[n - 1, 0] = 0
    flat = torch.zeros(off + n * ld, dtype=torch.from_numpy(D).dtype).pin_memory()
    Dh = flat[off:].view(n, ld)
    Dh[:, :S] = torch.from_numpy(D)
    want, wsum, winf, _ = oracle.split_costs(inst.tour, inst.dist, D, inst.Q, inst.L, nthreads=8)
    sp = cv.Splitter(0)
    out = torch.full((S,), -7, dtype=torch.int32).pin_memory()
    for _ in range(2):                                       # the second call finds the first one's totals
        r = sp.split_host(inst.tour, inst.dist, Dh, inst.Q, inst.L, S=S, out_cost=out)
        assert np.array_equal(out.numpy(), want)
        assert (r.sum, r.infeasible) == (wsum, winf)
    dev = torch.empty(S, dtype=torch.int32, device="cuda")
    sp.split(inst.tour, inst.dist, torch.from_numpy(D).cuda(), inst.Q, inst.L, out_cost=dev)
    assert np.array_equal(out.numpy(), dev.cpu().numpy())
    sp.close()


def test_staged_rows_set_aside(cv):
    """Customers ever farther from the depot: 27 to 29 candidates stay in the
    deque, the ring of 16 overflows and the second pass evaluates the scenarios."""
    n, S = 90, 24577
    inst = make_instance(n, 5, 30, 8, Q=400, L=n)
    ang = np.argsort(np.random.default_rng(1).permutation(n))
    pts = np.vstack([[0.0, 0.0], np.stack([1000 + 10.0 * np.arange(n), 3.0 * ang], 1)])
    dist = np.rint(np.hypot(*(pts[:, None] - pts[None]).transpose(2, 0, 1))).astype(np.int32)
    tour = np.arange(1, n + 1, dtype=np.int32)
    D = np.random.default_rng(2).integers(0, 12, (n, S)).astype(np.int16)
    want, wsum, winf, _ = oracle.split_costs(tour, dist, D, inst.Q, n, nthreads=8)
    sp = cv.Splitter(0)
    out = torch.empty(S, dtype=torch.int32).pin_memory()
    r = sp.split_host(tour, dist, torch.from_numpy(D).pin_memory(), inst.Q, n, out_cost=out)
    assert sp.stats()["overflow"] > S // 2
    assert np.array_equal(out.numpy(), want)
    assert (r.sum, r.infeasible) == (wsum, winf)
    sp.close()
