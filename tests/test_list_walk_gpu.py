"""Long lists of set-aside scenarios: rings of 16 overflow, the second pass
walks the list with rings of 32, and what that cannot settle (deques longer
still, negative demands) goes to the warp kernel. Against the oracle, bit for
bit, beside infeasible scenarios, in both types, from device and host memory."""
import numpy as np
import pytest

import oracle
from synth import make_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

S = 140_000                                  # rings of 16, also on devices of 152 SMs


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


# windows of about 24 (all settled by rings of 32), of 24 and 48, of 48 (none settled)
@pytest.mark.parametrize("windows", ["24", "both", "48"])
@pytest.mark.parametrize("cap", [False, True])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_long_lists(cv, windows, cap, dtype):
    n, Q, L = 70, 240, 21 if cap else 70
    tour, dist = growing(n)
    rng = np.random.default_rng([n, len(windows), cap])
    D = rng.integers(9, 12, (n, S)).astype(dtype)
    if windows != "24":
        D[:, (slice(None) if windows == "48" else slice(S // 3, None))] //= 2
    D[n // 2, 5::1000] = Q + 1
    D[0, 7] = 32767
    want, ws, wi, _ = oracle.split_costs(tour, dist, D, Q, L, nthreads=8)
    sp = cv.Splitter(0)
    dev, out = torch.from_numpy(D).cuda(), torch.empty(S, dtype=torch.int32, device="cuda")
    for _ in range(2):                       # the second call finds the first one's totals
        r = sp.split(tour, dist, dev, Q, L, out_cost=out)
        assert sp.stats()["ring"] == 16 and sp.stats()["overflow"] > S // 2
        assert np.array_equal(out.cpu().numpy(), want)
        assert (r.sum, r.infeasible) == (ws, wi) and wi == S // 1000 + 1
    host = torch.empty(S, dtype=torch.int32).pin_memory()
    r = sp.split_host(tour, dist, torch.from_numpy(D).pin_memory(), Q, L, out_cost=host)
    assert np.array_equal(host.numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    dev[3, S - 2] = -1
    with pytest.raises(cv.CvrpsdError):
        sp.split(tour, dist, dev, Q, L, out_cost=out)
    with pytest.raises(cv.CvrpsdError):
        sp.check_inputs()
    sp.check_inputs()
    sp.close()


@pytest.mark.parametrize("extra", [-1, 0, 1])               # around the list's length from which it is walked
def test_line_between_the_passes(cv, extra):
    n, Q, listed = 40, 240, 16384 + extra
    tour, dist = growing(n)
    D = np.full((n, S), 60, np.int16)        # windows of 4
    D[:, :listed] = 10
    want, ws, wi, _ = oracle.split_costs(tour, dist, D, Q, n, nthreads=8)
    sp = cv.Splitter(0)
    out = torch.empty(S, dtype=torch.int32, device="cuda")
    r = sp.split(tour, dist, torch.from_numpy(D).cuda(), Q, n, out_cost=out)
    assert sp.stats()["overflow"] == listed and sp.stats()["launches"] == 2
    assert np.array_equal(out.cpu().numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    sp.close()
