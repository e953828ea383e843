"""The warp kernel's register walk (windows of up to 64 candidates in two
registers per lane, four positions to a step, 32 to a chunk) and its hand-over
of longer windows, against the oracle, bit for bit: tour lengths around the
step, chunk and register edges, window lengths from one position to past 64."""
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


def split(cv, sp, inst, D, Q, L):
    out = torch.full((D.shape[1],), -5, dtype=torch.int32, device="cuda")
    r = sp.split(inst.tour, inst.dist, torch.from_numpy(D).cuda(), Q, L, out_cost=out)
    return r, out.cpu().numpy()


@pytest.mark.parametrize("n", [1, 4, 5, 31, 32, 33, 64, 65, 66, 97, 130, 261])
@pytest.mark.parametrize("Q", [9, 60, 210, 420, 5000])       # windows of about 2, 11, 38, 76 and all positions
@pytest.mark.parametrize("L", [3, 33, 64, 10_000])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_windows_and_tour_lengths(cv, n, Q, L, dtype):
    rng = np.random.default_rng([n, Q, L])
    inst = make_instance(n, 1, 10, seed=n, Q=Q, L=L)
    D = rng.integers(0, 10, size=(n, 67)).astype(dtype)
    D[:, 1] = 0                                  # every window as long as L allows
    D[rng.integers(0, n), 2] = Q + 1             # infeasible
    D[n - 1, 3] = 32767 if Q < 32767 else Q
    sp = cv.Splitter(0)
    sp.configure(kernel=cv.KERNEL_WARP)
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, min(L, n), nthreads=4)
    r, got = split(cv, sp, inst, D, Q, L)
    assert np.array_equal(got, want)
    assert (r.sum, r.infeasible) == (ws, wi) and wi >= 2
    assert sp.stats()["kernel"] == cv.KERNEL_WARP
    D[n // 2, 4] = -1                            # reported, also behind a demand above Q
    if n > 1:
        D[0, 4] = Q + 1
    with pytest.raises(cv.CvrpsdError):
        split(cv, sp, inst, D, Q, L)
    with pytest.raises(cv.CvrpsdError):
        sp.check_inputs()
    sp.check_inputs()
    sp.close()


@pytest.mark.parametrize("S", [1, 48, 49, 8192, 8193])
@pytest.mark.parametrize("n", [63, 64, 899, 900])
def test_automatic_choice_is_exact(cv, n, S):
    rng = np.random.default_rng([n, S])
    inst = make_instance(n, 1, 30, seed=n + S, Q=200, L=60)
    D = rng.integers(1, 31, size=(n, S)).astype(np.int16)
    sp = cv.Splitter(0)
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, 200, 60, nthreads=8)
    r, got = split(cv, sp, inst, D, 200, 60)
    assert np.array_equal(got, want) and (r.sum, r.infeasible) == (ws, wi)
    sp.close()


@pytest.mark.parametrize("more", [-1, 0, 1])                 # around four scenarios per SM: pairs, then lone warps
@pytest.mark.parametrize("n,Q", [(1, 30), (32, 60), (33, 60), (200, 150), (200, 700)])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_pairs_and_lone_warps(cv, more, n, Q, dtype):
    S = 4 * torch.cuda.get_device_properties(0).multi_processor_count + more
    rng = np.random.default_rng([n, S])
    inst = make_instance(n, 1, 10, seed=n + S, Q=Q)
    D = rng.integers(0, 20, size=(n, S)).astype(dtype)
    D[:, 1] = 0                                              # a window of the whole tour, after short ones
    D[: n // 2, 2] = 5
    D[n // 2:, 2] = 0
    D[n - 1, 3] = Q + 1
    D[0, S - 1] = Q + 1
    sp = cv.Splitter(0)
    sp.configure(kernel=cv.KERNEL_WARP)
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, n, nthreads=4)
    for _ in range(2):                                       # the second call finds the first one's totals
        r, got = split(cv, sp, inst, D, Q, n)
        assert np.array_equal(got, want)
        assert (r.sum, r.infeasible) == (ws, wi) and wi >= 2
    D[0, 3] = -1                                             # beside a demand above Q (n = 1: alone)
    with pytest.raises(cv.CvrpsdError):
        split(cv, sp, inst, D, Q, n)
    sp.close()


@pytest.mark.parametrize("n,S", [(2999, 48), (3000, 48), (3000, 49)])
def test_automatic_choice_of_long_tours_is_exact(cv, n, S):
    test_automatic_choice_is_exact(cv, n, S)


def test_calls_without_a_stream_take_the_current_one(cv):
    s = torch.cuda.Stream()
    assert cv._stream_ptr(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(s):
        assert cv._stream_ptr(None) == s.cuda_stream
    assert cv._stream_ptr(s) == s.cuda_stream and cv._stream_ptr(7) == 7
