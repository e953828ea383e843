"""Large means, whose entries the generator evaluates in float64 throughout: every
entry is the float64 recipe's where both ways are in one matrix, and correlated
entries cost no second normal each."""
import numpy as np
import pytest

from test_gen_f64_gpu import recipe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv():
    from paper_2511_18022_gb300 import build
    build.build()
    import paper_2511_18022_gb300 as m
    return m


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("bits", [16, 32])
# blocks of 8 rows and of 64 (their last one partly filled), means around both lines, mixed and all above
@pytest.mark.parametrize("n,S,lo,hi", [(1, 1, 2**31 - 1, 2**31 - 1), (9, 257, 87_499, 87_501), (131, 4097, 1, 200_000),
                                       (70, 80_001, 10_900, 11_000), (70, 80_001, 99_990, 100_010),
                                       (65, 40_000, 200_000, 2_000_000)])
def test_every_entry_is_the_float64_recipe(cv, kind, bits, n, S, lo, hi):
    rng = np.random.default_rng([kind, bits, n, lo])
    mu = rng.integers(lo, hi + 1, n).astype(np.int32)
    region = rng.integers(0, 4, n).astype(np.int32)
    seed = int(rng.integers(0, 1 << 63))
    sp = cv.Splitter(0)
    out = torch.full((n, S + 3), -7, dtype=torch.int16 if bits == 16 else torch.int32, device="cuda")
    sp.gen_demand(seed, kind, mu, region, out, S=S)
    want = recipe(seed, kind, mu, region, S, 32767 if bits == 16 else 2**31 - 1)
    assert torch.equal(out[:, :S].to(torch.float64), want)
    assert bool((out[:, S:] == -7).all())
    sp.close()


def test_correlated_entries_share_their_factors(cv):
    """Time of a correlated matrix over that of a normal one: one normal and an
    exponential an entry give 1.3; a second normal for each gave 2.0."""
    n, S = 200, 100_000
    mu, region = np.full(n, 1_000_000, np.int32), np.arange(n, dtype=np.int32) % 4
    out, sp = torch.empty((n, S), dtype=torch.int32, device="cuda"), cv.Splitter(0)
    ms = {0: [], 1: []}
    for rep in range(6):
        for kind in (0, 1):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sp.gen_demand(rep, kind, mu, region, out)
            b.record()
            torch.cuda.synchronize()
            ms[kind].append(a.elapsed_time(b))
    assert min(ms[1]) < 1.6 * min(ms[0])
    sp.close()
