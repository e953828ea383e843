"""What a waiting call with set-aside scenarios puts on the stream: the main
kernel, the table that the pass over the list reads, and that pass, which hands
its totals to the host and clears them itself."""
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


def on_stream(call):
    """Names of the copies, memsets and kernels of one call, in order."""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):                                       # a process's first profile may come up empty
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            call()
            torch.cuda.synchronize()
        ev = [e for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA]
        if ev:
            break
    return [e.name for e in sorted(ev, key=lambda e: e.time_range.start)]


@pytest.mark.parametrize("n,S,listed", [(30, 500, 1), (30, 500, 7), (80, 9001, 3), (80, 9001, 9001), (200, 8193, 5000)])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_one_pass_and_no_copies_back(cv, n, S, listed, dtype):
    Q = 90
    inst = make_instance(n, 1, 10, seed=n, Q=Q)
    D = np.random.default_rng([n, listed]).integers(1, 20, (n, S)).astype(dtype)
    D[n // 2, :listed] = Q + 1
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, Q, n, nthreads=8)
    sp = cv.Splitter(0)
    dev, out = torch.from_numpy(D).cuda(), torch.empty(S, dtype=torch.int32, device="cuda")
    results = []

    def call():
        results.append(sp.split(inst.tour, inst.dist, dev, Q, n, out_cost=out))

    for _ in range(2):                                       # the second call finds the first one's totals
        call()
    names = on_stream(call)
    assert sp.stats()["overflow"] == listed and sp.stats()["launches"] == 2
    assert np.array_equal(out.cpu().numpy(), want)
    assert all((r.sum, r.infeasible) == (ws, wi) for r in results) and wi == listed
    assert not any("DtoH" in k or "Memset" in k for k in names), names
    assert sum("split" in k for k in names) == 2 and sum("HtoD" in k for k in names) == 1, names
    bad = dev.clone()
    bad[0, 0] = -1
    with pytest.raises(cv.CvrpsdError):
        sp.split(inst.tour, inst.dist, bad, Q, n)
    r = sp.split(inst.tour, inst.dist, dev, Q, n, out_cost=out)
    assert (r.sum, r.infeasible) == (ws, wi)
    sp.close()
