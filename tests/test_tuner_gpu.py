"""The tuner against the library's own choice: what it keeps must not be slower
on the workload it timed, nor bind calls of other kinds where it found nothing
better, and a shape it may keep has to be the one that runs."""
import json

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


def strips(n, S):
    """A tour in strips: rings of 16 set scenarios aside, rings of 32 do not."""
    inst = make_instance(n, 5, 20, seed=3, Q=150)
    xy = inst.coords[inst.tour]
    inst.tour = inst.tour[np.lexsort((xy[:, 0], xy[:, 1] * 6 // (xy[:, 1].max() + 1)))].copy()
    D = np.random.default_rng(n).integers(2, 19, (n, S)).astype(np.int16)
    return inst, D


@pytest.mark.parametrize("S,ring", [(100_000, 32), (3000, None)])
def test_own_choice_is_kept_where_no_shape_beats_it(cv, tmp_path, S, ring):
    inst, D = strips(200, S)
    dev, cache = torch.from_numpy(D).cuda(), tmp_path / "tune.jsonl"
    sp = cv.Splitter(0)
    t = sp.autotune(inst.tour, inst.dist, dev, inst.Q, inst.n, cache_path=cache)
    assert (t["threads"], t["spt"], t["ring"]) == (0, 0, 0) and t["ms"] > 0
    assert json.loads(cache.read_text())["threads"] == 0
    again = sp.autotune(inst.tour, inst.dist, dev, inst.Q, inst.n, cache_path=cache)
    assert again["shapes_timed"] == 0 and again["threads"] == 0
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, inst.Q, inst.n, nthreads=8)
    r = sp.split(inst.tour, inst.dist, dev, inst.Q, inst.n)
    st = sp.stats()
    assert (r.sum, r.infeasible) == (ws, wi) and st["overflow"] == 0
    assert st["ring"] == ring if ring else st["kernel"] == cv.KERNEL_WARP
    sp.split(inst.tour, inst.dist, dev, inst.Q, inst.n, S=40)
    assert sp.stats()["kernel"] == cv.KERNEL_WARP            # not the kernel of a forced shape
    sp.close()


@pytest.mark.parametrize("rounds", [0, 3])
def test_rings_of_32_on_request(cv, rounds):
    inst, D = strips(120, 10_001)
    want, ws, wi, _ = oracle.split_costs(inst.tour, inst.dist, D, inst.Q, inst.n, nthreads=8)
    sp = cv.Splitter(0)
    sp.configure(kernel=cv.KERNEL_DEQUE, threads=64, spt=1, ring=32, variant=cv.WALK_PARAM_TABLE, rounds=rounds)
    out = torch.empty(D.shape[1], dtype=torch.int32, device="cuda")
    r = sp.split(inst.tour, inst.dist, torch.from_numpy(D).cuda(), inst.Q, inst.n, out_cost=out)
    st = sp.stats()
    assert (st["variant"], st["threads"], st["ring"], st["rounds"]) == (cv.WALK_PARAM_TABLE, 64, 32, rounds)
    assert np.array_equal(out.cpu().numpy(), want) and (r.sum, r.infeasible) == (ws, wi)
    sp.close()
