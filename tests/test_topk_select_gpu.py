"""Top-k by selection (k up to 1024) and by the full sort (k above), against
numpy: scores that share leading bits, many equal ones, NaN and infinities, and
every score wanted."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def expected(s, k):
    order = sorted(range(len(s)), key=lambda i: (bool(np.isnan(s[i])), 0.0 if np.isnan(s[i]) else s[i], i))
    return np.array(order[:k], np.int32)


@pytest.mark.parametrize("M,k", [(1, 1), (33, 33), (1000, 1), (1024, 1024), (1025, 1024), (4096, 64), (5000, 1025),
                                 (16384, 777), (16384, 16384)])
@pytest.mark.parametrize("kind", ["normal", "near", "equal", "few", "special"])
def test_topk(M, k, kind):
    import paper_2511_18022_gb300 as cv
    from paper_2511_18022_gb300 import build
    build.build()
    rng = np.random.default_rng([M, k])
    s = rng.normal(size=M).astype(np.float32)
    if kind == "near":
        s = (1.0 + 1e-6 * s).astype(np.float32)
    elif kind == "equal":
        s[:] = -3.5
    elif kind == "few":
        s = rng.integers(-2, 3, M).astype(np.float32)
    elif kind == "special":
        s[rng.random(M) < 0.3] = np.nan
        s[rng.random(M) < 0.1] = np.inf
        s[rng.random(M) < 0.1] = -np.inf
    sp = cv.Splitter(0)
    out = torch.full((k,), -1, dtype=torch.int32, device="cuda")
    cv.cvrpsd_topk(sp.ctx, torch.from_numpy(s).cuda(), k, out)
    assert np.array_equal(out.cpu().numpy(), expected(s, k))
    sp.close()
