"""Rings of 32 in the parameter-table walk's own choice: blocks of 64 threads, of
448 for the last scenarios that an SM's shared memory holds, and rings of 16
beyond, at the sizes from which the blocks no longer fit the device at once; each
shape has to equal the oracle bit for bit, with predecessors too."""
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


def resident(threads):
    """Scenarios the device holds: rings of 32 entries of 8 bytes, 512 bytes of sums, 1 KB a block for the system."""
    p = torch.cuda.get_device_properties(0)
    return p.shared_memory_per_multiprocessor // (threads * 32 * 8 + 512 + 1024) * threads * p.multi_processor_count


@pytest.mark.parametrize("kind", ["random", "smooth", "growing"])
@pytest.mark.parametrize("threads,more,want_shape", [(64, 0, (64, 32)), (64, 1, (448, 32)), (448, 0, (448, 32)),
                                                     (448, 1, (128, 16))])
@pytest.mark.parametrize("cap", [False, True])
def test_shape_and_costs(cv, kind, threads, more, want_shape, cap):
    n, Q = 41, 200
    S = resident(threads) + more
    inst = make_instance(n, 1, 10, seed=n, Q=Q)
    if kind == "smooth":
        xy = inst.coords[inst.tour]
        inst.tour = inst.tour[np.lexsort((xy[:, 0], xy[:, 1] * 3 // (xy[:, 1].max() + 1)))].copy()
    if kind == "growing":                                    # every candidate stays in the deque
        pts = np.vstack([[0.0, 0.0], np.stack([1000 + 10.0 * np.arange(n), np.full(n, 200.0)], 1)])
        inst.dist = np.rint(np.hypot(*(pts[:, None] - pts[None]).transpose(2, 0, 1))).astype(np.int32)
        inst.tour = np.arange(1, n + 1, dtype=np.int32)
    L = 30 if cap else n
    D = np.random.default_rng([n, S]).integers(0, 20, (n, S)).astype(np.int16)
    D[:, 1::97] //= 4                                        # deques of 30 and more on the growing tour
    D[n // 2, 2::501] = Q + 1
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, L, nthreads=8)
    sp = cv.Splitter(0)
    dev, out = torch.from_numpy(D).cuda(), torch.empty(S, dtype=torch.int32, device="cuda")
    r = sp.split(inst.tour, inst.dist, dev, Q, L, out_cost=out)
    st = sp.stats()
    assert (st["threads"], st["ring"]) == want_shape
    assert np.array_equal(out.cpu().numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    pred = torch.empty((n, S), dtype=torch.int16, device="cuda")
    r = sp.split_routes(inst.tour, inst.dist, dev, Q, L, pred=pred, out_cost=out)
    st = sp.stats()
    assert (st["threads"], st["ring"]) == want_shape
    assert np.array_equal(out.cpu().numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    for s in (0, 1, S // 2, S - 1):
        cost, _, opred = oracle.split_routes(inst.tour, inst.dist, D[:, s], Q, L)
        assert cost is None or np.array_equal(pred[:, s].cpu().numpy(), opred[1:]), f"scenario {s}"
    sp.close()
