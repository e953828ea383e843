"""Windows of more than 64 positions in the register walk: the values of older
positions come from rings in shared memory. Against the oracle, bit for bit, at
tour lengths around chunk and ring edges, windows from a few positions to the
whole tour in one call, and on both sides of the lines of the automatic choice,
which takes the walk only where it holds every window that n and L allow."""
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


def demands(n, S, Q, dtype, seed):
    """Scenarios of long, short and mixed windows: a load per column, some of
    zeros, some that change along the tour, some infeasible."""
    rng = np.random.default_rng(seed)
    D = (rng.integers(0, 20, (n, S)) * rng.choice([0, 1, 1, 4, 40], S) // 4).astype(dtype)
    D[: n // 2, 1] = 0
    D[n // 3: n // 2, 2] = min(Q, 32767) // 3                # windows of 3 between long ones
    D[::7, 3] = min(Q, 32767)
    D[n - 1, S // 2] = min(Q + 1, 32767)
    return D


def check(cv, sp, inst, D, Q, L, **kw):
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, L, nthreads=8)
    out = torch.full((D.shape[1],), -5, dtype=torch.int32, device="cuda")
    r = sp.split(inst.tour, inst.dist, torch.from_numpy(D).cuda(), Q, L, out_cost=out, **kw)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), want)
    if kw.get("host_outputs", True):
        assert (r.sum, r.infeasible) == (ws, wi)
    return sp.stats()


# tours of up to a whole ring (no slot used twice) and longer ones under a route
# length that keeps the ring short; pairs of warps (67 scenarios) and lone warps
@pytest.mark.parametrize("S", [67, 700])
@pytest.mark.parametrize("n,L", [(65, 65), (66, 66), (96, 96), (97, 97), (129, 129), (191, 65), (257, 64), (300, 100),
                                 (450, 193), (700, 192), (1000, 1000), (1100, 449)])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_far_windows(cv, n, L, S, dtype):
    Q = 9 * n
    inst = make_instance(n, 1, 10, seed=n + L, Q=Q, L=L)
    D = demands(n, S, Q, dtype, [n, L, S])
    sp = cv.Splitter(0)
    for wait in (True, False, True):
        st = check(cv, sp, inst, D, Q, L, host_outputs=wait)
        assert st["kernel"] == cv.KERNEL_WARP and (not wait or st["overflow"] == 0)
    D[n // 2, 4] = -1
    with pytest.raises(cv.CvrpsdError):
        sp.split(inst.tour, inst.dist, torch.from_numpy(D).cuda(), Q, L)
    sp.close()


# the automatic choice: up to 8192 scenarios from 64 positions on, the sequence-parallel
# kernel for up to 48 from 3000 on, and neither where the walk's rings are too short
@pytest.mark.parametrize("n,S,L,kernel", [
    (63, 700, 63, 1), (64, 700, 64, 2), (100, 8192, 100, 2), (100, 8193, 100, 1), (900, 1, 900, 2),
    (2999, 48, 60, 2), (3000, 48, 60, 3), (3000, 49, 60, 2), (3000, 49, 3000, 2), (3000, 700, 3000, 2),
    (3000, 2000, 3000, 1), (3000, 2000, 300, 2), (8000, 500, 8000, 1), (8000, 200, 8000, 2)])
def test_automatic_choice(cv, n, S, L, kernel):
    Q = 5 * min(n, 2 * L)
    inst = make_instance(n, 1, 10, seed=n + S, Q=Q, L=L)
    D = np.random.default_rng([n, S]).integers(0, 21, (n, S)).astype(np.int16)
    sp = cv.Splitter(0)
    st = check(cv, sp, inst, D, Q, L)
    assert st["kernel"] == kernel and (kernel != cv.KERNEL_WARP or st["overflow"] == 0)
    sp.close()


def test_forced_walk_sets_longer_windows_aside(cv):
    """More scenarios than leave room for rings of a whole tour."""
    n, S = 3000, 2000
    inst = make_instance(n, 1, 10, seed=4, Q=10 * n)
    D = np.random.default_rng(7).integers(0, 9, (n, S)).astype(np.int16)
    D[:, ::2] *= 100
    sp = cv.Splitter(0)
    sp.configure(kernel=cv.KERNEL_WARP)
    st = check(cv, sp, inst, D, 10 * n, n)
    assert st["kernel"] == cv.KERNEL_WARP and 0 < st["overflow"] < S
    sp.close()
