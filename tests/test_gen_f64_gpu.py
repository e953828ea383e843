"""The generator decides most entries in float32 and the rest in float64; every
entry has to be the float64 recipe's. Reference: the recipe in torch float64
operations on the GPU (each rounded on its own) over host Philox words. Exact
equality is asked for: an entry can only differ where the two float64
evaluations, an ulp apart, straddle a rounding boundary (about 1e-14)."""
import numpy as np
import pytest

from synth.rng import philox4x32_10

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def normal(s, index, domain, seed):
    w = philox4x32_10(s[None, :], index[:, None], domain, 0, seed & 0xFFFFFFFF, seed >> 32)
    u1 = (torch.from_numpy(w[0].astype(np.float64)).cuda() + 0.5) * 2.0 ** -32
    u2 = torch.from_numpy(w[1].astype(np.float64)).cuda() * 2.0 ** -32
    return torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(6.283185307179586 * u2)


def recipe(seed, kind, mu, region, S, top):
    s, rows = np.arange(S, dtype=np.int64), np.arange(len(mu), dtype=np.int64)
    m = torch.from_numpy(mu.astype(np.float64)).cuda()[:, None]
    if kind == 1:
        f = normal(s, np.arange(4), 1, seed)[torch.from_numpy(region.astype(np.int64)).cuda()]
        y = 0.6 * f + 0.8 * normal(s, rows, 0, seed)
        x = m * torch.exp(0.3 * y - 0.045)
    else:
        x = m + (0.3 * m) * normal(s, rows, 2, seed)
    r = torch.floor(x)
    return (r + (x - r >= 0.5)).clamp(0, top)


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("mu_hi", [0, 30, 3000, 60_000, 30_000_000])   # 30: all in float32; the last: all in float64
@pytest.mark.parametrize("n,S", [(1, 1), (65, 255), (131, 4097)])
def test_every_entry_is_the_float64_recipe(kind, bits, mu_hi, n, S):
    import paper_2511_18022_gb300 as cv
    from paper_2511_18022_gb300 import build
    build.build()
    rng = np.random.default_rng([kind, bits, mu_hi, n])
    mu = rng.integers(0, mu_hi + 1, n).astype(np.int32)
    region = rng.integers(0, 4, n).astype(np.int32)
    seed = int(rng.integers(0, 1 << 63))
    sp = cv.Splitter(0)
    out = torch.full((n, S + 3), -7, dtype=torch.int16 if bits == 16 else torch.int32, device="cuda")
    sp.gen_demand(seed, kind, mu, region, out, S=S)
    want = recipe(seed, kind, mu, region, S, 32767 if bits == 16 else 2**31 - 1)
    assert torch.equal(out[:, :S].to(torch.float64), want)
    assert bool((out[:, S:] == -7).all())
    sp.close()
