"""stats()['launches'] is the number of kernels that a call put on its stream."""
import numpy as np
import pytest

from synth import make_instance
from test_aside_trip_gpu import on_stream

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cv():
    from paper_2511_18022_gb300 import build
    build.build()
    import paper_2511_18022_gb300 as m
    return m


# blocks of 64 and 128 threads, which have one walk, of 512 and 256, which have two, and
# capacities whose keys the second walk cannot hold
@pytest.mark.parametrize("n,T,S,Q,threads,launches", [(60, 4, 100, 100, 64, 4), (400, 64, 3000, 100, 128, 4),
                                                     (700, 64, 9000, 100, 512, 5), (2000, 16, 20_000, 100, 256, 5),
                                                     (65, 64, 9000, 1_000_000, 256, 4)])
def test_tours_of_one_instance(cv, n, T, S, Q, threads, launches):
    rng = np.random.default_rng(n)
    inst = make_instance(n, 1, 10, seed=3, Q=Q)
    tours = torch.from_numpy(np.stack([rng.permutation(n) + 1 for _ in range(T)]).astype(np.int32)).cuda()
    D = torch.from_numpy(rng.integers(1, 11, (n, S)).astype(np.int32 if Q > 32767 else np.int16)).cuda()
    mean = torch.empty(T, dtype=torch.float64, device="cuda")
    sp = cv.Splitter(0)

    def call():
        cv.cvrpsd_split_eval_tours(sp.ctx, tours, inst.dist, D, Q, mean=mean)

    call()
    names = on_stream(call)
    st = sp.stats()
    assert (st["threads"], st["launches"]) == (threads, launches)
    assert sum("kernel" in k for k in names) == launches, names
    sp.close()


@pytest.mark.parametrize("n,S,kernel,launches", [(100, 40, 2, 3), (50, 300, 1, 3), (4081, 60, 2, 5), (3000, 9, 3, 6)])
def test_recorded_calls(cv, n, S, kernel, launches):
    """Into a graph the tour table goes by kernels of up to 2040 entries each."""
    inst = make_instance(n, 1, 10, seed=4, Q=60, L=60)
    D = torch.from_numpy(np.random.default_rng(n).integers(1, 11, (n, S)).astype(np.int16)).cuda()
    sp, s = cv.Splitter(0), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        sp.split(inst.tour, inst.dist, D, 60, 60)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        sp.split(inst.tour, inst.dist, D, 60, 60, host_outputs=False)
    st = sp.stats()
    names = on_stream(g.replay)
    assert st["kernel"] == kernel
    assert st["launches"] == sum("kernel" in k for k in names) == launches, names
    sp.close()
