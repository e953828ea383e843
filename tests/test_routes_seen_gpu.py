"""Which kernel serves scenarios in host memory, on both sides of the staged walk's
lines, and recorded calls of the shapes that take opted-in shared memory."""
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


# (S, pitch, bytes before the matrix): staged from 24,576 scenarios on, where rows
# straddle 64-byte lines and the matrix starts on 16 bytes
@pytest.mark.parametrize("S,ld,before,staged", [
    (24_575, 24_577, 0, False), (24_576, 24_577, 0, True), (24_576, 24_576, 0, False), (24_576, 24_576, 16, True),
    (24_576, 24_608, 64, False), (30_000, 30_001, 4, False), (30_000, 30_001, 48, True), (40_001, 40_032, 0, False)])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_staged_walk(cv, S, ld, before, staged, dtype):
    n, Q, size = 23, 90, np.dtype(dtype).itemsize
    inst = make_instance(n, 1, 10, seed=2, Q=Q)
    D = np.random.default_rng(S).integers(0, 20, (n, S)).astype(dtype)
    flat = torch.zeros(before // size + n * ld + 64, dtype=torch.from_numpy(D).dtype).pin_memory()
    start = before // size + (-flat.data_ptr() % 64) // size
    Dh = flat[start: start + n * ld].view(n, ld)
    Dh[:, :S] = torch.from_numpy(D)
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, n, nthreads=8)
    sp, out = cv.Splitter(0), torch.empty(S, dtype=torch.int32).pin_memory()
    r = sp.split_host(inst.tour, inst.dist, Dh, Q, n, S=S, out_cost=out)
    assert sp.stats()["threads"] == (1024 // size if staged else 128)
    assert np.array_equal(out.numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    sp.close()


@pytest.mark.parametrize("n,S,kernel,shape", [(4000, 60, 2, None), (1000, 700, 2, None), (45, 130_000, 1, (448, 32))])
def test_recorded_calls(cv, n, S, kernel, shape):
    Q = 9 * n
    rec, other = (make_instance(n, 1, 10, seed=s, Q=Q) for s in (1, 2))
    D = np.random.default_rng(n).integers(0, 20, (n, S)).astype(np.int16)
    want = oracle.split_costs(rec.tour, rec.dist, D, Q, n, nthreads=8)[0]
    sp, s, dev, out = cv.Splitter(0), torch.cuda.Stream(), torch.from_numpy(D).cuda(), torch.empty(S, dtype=torch.int32,
                                                                                                     device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        sp.split(rec.tour, rec.dist, dev, Q)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        sp.split(rec.tour, rec.dist, dev, Q, out_cost=out, host_outputs=False)
    st = sp.stats()
    assert st["kernel"] == kernel and (shape is None or (st["threads"], st["ring"]) == shape)
    with torch.cuda.stream(s):
        sp.split(other.tour, other.dist, dev, Q)
        g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), want)
    sp.close()
