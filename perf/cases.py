"""The work that users have this library do, as measurable cases.

Every case is one pass through the public entry points (the `Splitter`
methods, the batch, the local search and the surrogate network) on inputs of
the shapes the library is used with. Instances are synthetic as everywhere in
this repository: customers uniform on a 1000 x 1000 grid around a central
depot, rounded Euclidean distances, mean demands uniform integers, scenarios
normal (sd 0.3 of the mean) or lognormal with a factor per quadrant. Tours are
random permutations (what the workloads split and a search starts from) or
run through the customers in strips (what a search works on later: neighbours
in the tour are close together).

A case's "op" says which call it is:
  split    one tour under S scenarios, costs on the device, exact sums back
  routes   the same with the optimal predecessor of every position
  host     the same with the scenario matrix in page-locked host memory
  batch    many tours with their own scenarios, captured once, run again
  tours    candidate tours of one instance under one scenario matrix
  gen      the scenario generator
  predict  the surrogate's scores of candidate tours
  train    an epoch of the surrogate over mini-batches, then its checkpoint
  search   iterations of the screened local search
"""
import math

import numpy as np
import torch

import paper_2511_18022_gb300 as cv
from paper_2511_18022_gb300 import search as ls_mod

H, IN1, IN2 = 256, 5, 257                       # the surrogate's layer sizes
PARAMS = cv._lib.SURROGATE_PARAMS


def listed():
    return [
        # The small instance of the tests and the smoke run: one call of a user who
        # tries the library, or the inner loop of a search over few scenarios.
        {"name": "split-n50-S1000-i32", "op": "split", "n": 50, "S": 1000, "mu_lo": 1, "mu_hi": 10, "Q": 40,
         "L": 0, "i32": True, "corr": False, "strip": False},
        # A long tour under few scenarios: the call whose latency counts (an odd
        # number of scenarios, as a sample of a larger set has).
        {"name": "split-n1000-S37", "op": "split", "n": 1000, "S": 37, "mu_lo": 1, "mu_hi": 30, "Q": 200, "L": 60,
         "i32": False, "corr": True, "strip": False},
        # The ordinary evaluation: a middle-sized tour under 100,000 scenarios.
        {"name": "split-n200-S100000", "op": "split", "n": 200, "S": 100_000, "mu_lo": 5, "mu_hi": 20, "Q": 150,
         "L": 40, "i32": False, "corr": True, "strip": False},
        # The benchmark's headline workload: a large tour under 2^20 scenarios.
        {"name": "split-n1000-S1M", "op": "split", "n": 1000, "S": 1 << 20, "mu_lo": 1, "mu_hi": 30, "Q": 200,
         "L": 60, "i32": False, "corr": True, "strip": False},
        # Reading the routes off: the predecessors of a middle-sized tour.
        {"name": "routes-n200-S100000", "op": "routes", "n": 200, "S": 100_000, "mu_lo": 5, "mu_hi": 20, "Q": 150,
         "L": 40, "i32": False, "corr": True, "strip": False},
        # Scenarios that the user keeps in host memory (a ragged number of them).
        {"name": "host-n200-S99999", "op": "host", "n": 200, "S": 99_999, "mu_lo": 5, "mu_hi": 20, "Q": 150,
         "L": 40, "i32": False, "corr": True, "strip": False},
        # Many instances of 100 to 1000 customers at once, as the batched workload.
        {"name": "batch-T64-S8192", "op": "batch", "T": 64, "n_lo": 100, "n_hi": 1000, "S": 8192, "mu_lo": 1,
         "mu_hi": 10, "q_mult": 10, "corr": True},
        # The exact evaluation inside a search: the 64 best neighbours of a tour.
        {"name": "tours-T64-n200-S65536", "op": "tours", "T": 64, "n": 200, "S": 65_536, "mu_lo": 5, "mu_hi": 20,
         "Q": 150, "L": 40, "i32": False, "corr": True, "strip": True},
        # Making the scenario set of a workload.
        {"name": "gen-n200-S100000", "op": "gen", "n": 200, "S": 100_000, "mu_lo": 5, "mu_hi": 20, "i32": False,
         "corr": True},
        # Screening: the surrogate's scores of 4096 neighbours.
        {"name": "predict-T4096-n200", "op": "predict", "T": 4096, "n": 200, "strip": True},
        # Training: an epoch over 16 mini-batches of 1024 labelled tours.
        {"name": "train-B1024-n200", "op": "train", "T": 1024, "n": 200, "steps": 16, "strip": True},
        # The whole loop: 16 iterations of the screened local search.
        {"name": "search-M4096-n200", "op": "search", "n": 200, "S": 65_536, "mu_lo": 5, "mu_hi": 20, "Q": 150,
         "L": 40, "M": 4096, "k": 64, "iterations": 16, "corr": True, "strip": False},
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of lo..hi."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["split", "split", "split", "split", "routes", "host", "batch", "tours", "gen", "predict", "train",
                     "search"])
    corr = rng.random() < 0.7
    strip = rng.random() < 0.5
    i32 = rng.random() < 0.25
    mu_lo = rng.randint(1, 5)
    mu_hi = rng.randint(10, 30)
    Q = int((mu_lo + mu_hi) / 2 * rng.uniform(6, 16))
    L = 0 if rng.random() < 0.4 else rng.randint(20, 80)
    tour = {"mu_lo": mu_lo, "mu_hi": mu_hi, "Q": Q, "L": L, "i32": i32, "corr": corr, "strip": strip}
    if op == "split":
        n = _log_int(rng, 20, 1400)
        return {"op": op, "n": n, "S": _log_int(rng, 1, min(1 << 20, (1 << 28) // n)), **tour}
    if op in ("routes", "host"):
        n = _log_int(rng, 20, 1000)
        return {"op": op, "n": n, "S": _log_int(rng, 500, 20_000_000 // n), **tour}
    if op == "batch":
        T = _log_int(rng, 4, 64)
        n_lo = rng.randint(30, 300)
        return {"op": op, "T": T, "n_lo": n_lo, "n_hi": n_lo + rng.randint(10, 700), "S": _log_int(rng, 300, 8192),
                "mu_lo": 1, "mu_hi": 10, "q_mult": rng.randint(6, 14), "corr": corr}
    if op == "tours":
        n, T = _log_int(rng, 50, 500), _log_int(rng, 16, 128)
        return {"op": op, "T": T, "n": n, "S": _log_int(rng, 1000, min(65_536, 800_000_000 // (n * T))), **tour}
    if op == "gen":
        n = _log_int(rng, 20, 1000)
        return {"op": op, "n": n, "S": _log_int(rng, 500, 20_000_000 // n), "mu_lo": mu_lo, "mu_hi": mu_hi,
                "i32": i32, "corr": corr}
    if op == "predict":
        n = _log_int(rng, 50, 800)
        return {"op": op, "T": _log_int(rng, 64, min(8192, 1_600_000 // n)), "n": n, "strip": strip}
    if op == "train":
        n = _log_int(rng, 50, 500)
        return {"op": op, "T": _log_int(rng, 100, min(2048, 400_000 // n)), "n": n, "steps": rng.randint(4, 12),
                "strip": strip}
    n = _log_int(rng, 50, 300)
    return {"op": op, "n": n, "S": _log_int(rng, 2000, min(65_536, 8_000_000 // n)), "mu_lo": mu_lo, "mu_hi": mu_hi,
            "Q": Q, "L": L, "M": rng.randint(512, 4096), "k": rng.randint(16, 64), "iterations": rng.randint(4, 12),
            "corr": corr, "strip": strip}


# ---------------------------------------------------------------- inputs


class Inst:
    """One instance as the search module reads it."""

    def __init__(self, rng, n, mu_lo, mu_hi, Q, L, strip):
        self.n = n
        self.coords = np.vstack([[[500, 500]], rng.integers(0, 1001, (n, 2))]).astype(np.int64)
        d = self.coords.astype(np.float64)
        self.dist = np.floor(np.sqrt(((d[:, None, :] - d[None, :, :]) ** 2).sum(-1)) + 0.5).astype(np.int32)
        self.mu = rng.integers(mu_lo, mu_hi + 1, n).astype(np.int32)
        dx, dy = self.coords[1:, 0] - 500, self.coords[1:, 1] - 500
        self.region = ((dx < 0) + 2 * (dy < 0)).astype(np.int32)
        self.Q, self.L = int(Q), int(L or n)
        self.tour = self._strips() if strip else (rng.permutation(n) + 1).astype(np.int32)

    def _strips(self):
        """Customers in vertical strips, up one and down the next."""
        w = 1001.0 / max(1, int(math.sqrt(self.n / 2.0)))
        col = (self.coords[1:, 0] / w).astype(np.int64)
        y = np.where(col % 2 == 0, self.coords[1:, 1], -self.coords[1:, 1])
        return (np.lexsort((y, col)) + 1).astype(np.int32)


def _demands(inst, S, corr, i32, gen):
    """A [n][S] scenario matrix on the GPU, in blocks of rows."""
    dev = "cuda"
    D = torch.empty((inst.n, S), dtype=torch.int32 if i32 else torch.int16, device=dev)
    mu = torch.from_numpy(inst.mu).to(dev, torch.float32)[:, None]
    f = torch.randn((4, S), generator=gen, device=dev) if corr else None
    reg = torch.from_numpy(inst.region.astype(np.int64)).to(dev)
    rows = max(1, (1 << 26) // S)
    for a in range(0, inst.n, rows):
        b = min(inst.n, a + rows)
        x = torch.randn((b - a, S), generator=gen, device=dev)
        if corr:
            x.mul_(0.8).add_(f[reg[a:b]], alpha=0.6).mul_(0.3).sub_(0.045).exp_().mul_(mu[a:b])
        else:
            x.mul_(0.3).add_(1.0).mul_(mu[a:b])
        D[a:b] = x.round_().clamp_(0, 32767)
    return D


def _torch_gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _neighbours(rng, base, T):
    """T neighbours of a tour: a segment reversed or a customer moved."""
    n = len(base)
    out = np.tile(base, (T, 1))
    for t in range(1, T):
        a, b = sorted(int(v) for v in rng.integers(0, n, 2))
        if rng.integers(0, 2):
            out[t, a:b + 1] = base[a:b + 1][::-1]
        else:
            out[t, a:b + 1] = np.roll(base[a:b + 1], -1)
    return out.astype(np.int32)


def _params(rng):
    """Parameters of a network that has learned the obvious: the drawn weights, and an output that grows with the tour's length."""
    w1 = rng.uniform(-1, 1, (H, IN1)) / math.sqrt(IN1)
    b1 = rng.uniform(-1, 1, H) / math.sqrt(IN1)
    w2 = rng.uniform(-1, 1, (H, IN2)) / math.sqrt(IN2)
    b2 = rng.uniform(-1, 1, H) / math.sqrt(IN2)
    w3 = rng.uniform(-1, 1, H) / math.sqrt(H)
    w2[:, H] = np.sign(w3) * np.abs(w2[:, H]) * 4
    return np.concatenate([w1.ravel(), b1, w2.ravel(), b2, w3, [0.1]]).astype(np.float32)


def _net(rng, inst):
    """What the surrogate is built from: customer features, and the scale of its tour-length input."""
    mean = inst.mu * (1 + rng.normal(0, 0.01, inst.n))
    cust = np.column_stack([inst.coords[1:, 0], inst.coords[1:, 1], mean, 0.3 * mean]).astype(np.float32)
    return cust


def _lengths(tours, dist):
    t, d = tours.astype(np.int64), dist.astype(np.int64)
    return d[0, t[:, 0]] + d[t[:, -1], 0] + d[t[:, :-1], t[:, 1:]].sum(axis=1)


def _inputs(case, seed):
    """Everything of a case that is made from the seed alone."""
    rng = np.random.default_rng([seed, 77])
    op = case["op"]
    if op == "batch":
        insts = []
        for n in rng.integers(case["n_lo"], case["n_hi"] + 1, case["T"]):
            inst = Inst(rng, int(n), case["mu_lo"], case["mu_hi"], 1, 0, False)
            inst.Q = int(round(case["q_mult"] * float(inst.mu.mean())))
            insts.append(inst)
        gen = _torch_gen(seed)
        return insts, [_demands(i, case["S"], case["corr"], False, gen) for i in insts]
    if op in ("predict", "train"):
        inst = Inst(rng, case["n"], 5, 20, 150, 40, case["strip"])
        cust = _net(rng, inst)
        T = case["T"] * case.get("steps", 1)
        if op == "predict":
            tours = _neighbours(rng, inst.tour, T)
        else:
            tours = np.argsort(rng.random((T, case["n"])), axis=1).astype(np.int32) + 1
            tours[: T // 2] = _neighbours(rng, inst.tour, T // 2)
            tours = tours[rng.permutation(T)]
        lens = _lengths(tours, inst.dist).astype(np.float64)
        scale = (float(np.float32(lens.mean())), float(np.float32(lens.std() + 1.0)))
        target = ((lens - scale[0]) / scale[1] + 0.1 * rng.normal(0, 1, T)).astype(np.float32)
        p = _params(rng)
        m = (1e-3 * rng.normal(0, 1, PARAMS)).astype(np.float32)
        v = (1e-6 * rng.uniform(0.5, 1.5, PARAMS)).astype(np.float32)
        return inst, cust, tours, scale, target, p, m, v
    inst = Inst(rng, case["n"], case["mu_lo"], case["mu_hi"], case.get("Q", 1), case.get("L", 0),
                case.get("strip", False))
    if op == "gen":
        return inst, int(rng.integers(0, 1 << 62))
    D = _demands(inst, case["S"], case["corr"], case.get("i32", False), _torch_gen(seed))
    if op == "tours":
        return inst, D, _neighbours(rng, inst.tour, case["T"])
    if op == "search":
        return inst, D, _net(rng, inst), _params(rng), _neighbours(rng, inst.tour, 256)
    return inst, D


ADAM_STEP = 1000                                 # steps the resumed trainer has behind it
LR = 2e-4


class State(dict):
    """A user's handles, released in the order the library asks for: what was made on a context, then the context."""

    def __del__(self):
        for k in ("batch", "sur", "sp"):
            if k in self:
                self[k].close()


def prepare(case, seed):
    op = case["op"]
    x = _inputs(case, seed)
    sp = cv.Splitter(0)
    st = State(op=op, sp=sp, case=case)
    if op == "batch":
        insts, D = x
        outs = [torch.empty(case["S"], dtype=torch.int32, device="cuda") for _ in insts]
        st["tours"] = [{"tour": i.tour, "dist": i.dist, "demand": d, "Q": i.Q, "out_cost": o}
                       for i, d, o in zip(insts, D, outs)]
        st["outs"] = outs
        st["batch"] = sp.batch(st["tours"], case["S"])
        return st
    if op in ("predict", "train"):
        inst, cust, tours, scale, target, p, m, v = x
        sur = cv.Surrogate(sp.ctx, cust, inst.dist, inst.Q)
        sur.set_scale(*scale)
        st["sur"] = sur
        if op == "predict":
            sur.params(p)
            st["tours"] = torch.from_numpy(tours).cuda()
            st["out"] = torch.empty(case["T"], dtype=torch.float32, device="cuda")
            return st
        blob = bytearray(sur.state())            # 32-byte header, then parameters and Adam's moments
        np.frombuffer(blob, np.int32, 8)[4] = ADAM_STEP
        np.frombuffer(blob, np.float32, offset=32)[:] = np.concatenate([p, m, v])
        sur.load_state(bytes(blob))
        T = case["T"]
        st["batches"] = [(torch.from_numpy(tours[a:a + T]).cuda(), torch.from_numpy(target[a:a + T]).cuda())
                         for a in range(0, T * case["steps"], T)]
        st["loss"] = torch.zeros(case["steps"], dtype=torch.float32, device="cuda")
        return st
    inst = x[0]
    st["inst"] = inst
    if op == "gen":
        st["seed"] = x[1]
        st["out"] = torch.empty((case["n"], case["S"]), dtype=torch.int32 if case["i32"] else torch.int16,
                                device="cuda")
        return st
    st["D"] = x[1]
    if op == "tours":
        st["tours"] = torch.from_numpy(x[2]).cuda()
        st["mean"] = torch.empty(case["T"], dtype=torch.float64, device="cuda")
        st["sums"] = torch.empty(case["T"], dtype=torch.int64, device="cuda")
        st["inf"] = torch.empty(case["T"], dtype=torch.int64, device="cuda")
        return st
    if op == "search":
        sur = cv.Surrogate(sp.ctx, x[2], inst.dist, inst.Q)
        lens = _lengths(x[4], inst.dist)
        sur.set_scale(float(lens.mean()), float(lens.std() + 1.0))
        sur.params(x[3])
        st["sur"] = sur
        st["search"] = ls_mod.LocalSearch(sp.ctx, inst, x[1], inst.tour, surrogate=sur, M=case["M"], k=case["k"],
                                          seed=seed, moves_block=case["iterations"])
        return st
    if op == "host":
        D = torch.empty(x[1].shape, dtype=x[1].dtype, pin_memory=True)
        D.copy_(x[1])
        st["D"] = D
        st["out"] = torch.empty(case["S"], dtype=torch.int32, pin_memory=True)
        return st
    st["out"] = torch.empty(case["S"], dtype=torch.int32, device="cuda")
    if op == "routes":
        st["pred"] = torch.empty((case["n"], case["S"]), dtype=torch.int16, device="cuda")
    return st


# ---------------------------------------------------------------- the calls


def run(st):
    op, sp, case = st["op"], st["sp"], st["case"]
    if op == "batch":
        st["batch"].run()
        r = st["batch"].results()
        # at most a dozen of the per-tour cost vectors: outputs are limited in number
        return {"sum": r["sum"], "infeasible": r["infeasible"], "mean": r["mean"], "costs": st["outs"][:12]}
    if op == "gen":
        inst = st["inst"]
        sp.gen_demand(st["seed"], cv.GEN_CORRELATED if case["corr"] else cv.GEN_NORMAL, inst.mu, inst.region,
                      st["out"])
        return {"demand": st["out"]}
    if op == "predict":
        st["sur"].predict(st["tours"], st["out"])
        return {"scores": st["out"]}
    if op == "train":
        for k, (tours, target) in enumerate(st["batches"]):
            st["sur"].train_step(tours, target, LR, loss=st["loss"][k:k + 1])
        s = np.frombuffer(st["sur"].state(), np.float32, offset=32)
        return {"loss": st["loss"], "p": s[:PARAMS], "m": s[PARAMS:2 * PARAMS], "v": s[2 * PARAMS:]}
    inst = st["inst"]
    if op == "tours":
        cv.cvrpsd_split_eval_tours(sp.ctx, st["tours"], inst.dist, st["D"], inst.Q, inst.L, mean=st["mean"],
                                   sums=st["sums"], infeasible=st["inf"])
        return {"mean": st["mean"], "sum": st["sums"], "infeasible": st["inf"]}
    if op == "search":
        s = st["search"]
        s.run(case["iterations"])
        return {"tour": s.cur, "cost": s.cur_cost_t, "trace": np.array(s.log.costs[-case["iterations"]:])}
    if op == "routes":
        r = sp.split_routes(inst.tour, inst.dist, st["D"], inst.Q, inst.L, pred=st["pred"], out_cost=st["out"])
        return {"costs": st["out"], "pred": st["pred"], "sum": r.sum, "infeasible": r.infeasible, "mean": r.mean}
    call = sp.split_host if op == "host" else sp.split
    r = call(inst.tour, inst.dist, st["D"], inst.Q, inst.L, out_cost=st["out"])
    return {"costs": st["out"], "sum": r.sum, "infeasible": r.infeasible, "mean": r.mean}


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    """Bytes: each input read and each output written once. Operations: per (scenario, position) of a Split four
    (load, window test, minimum, cost); per generated demand ten Philox rounds and a Box-Muller draw, about 60;
    the network's multiply-adds, ReLU and pooling."""
    op = case["op"]
    if op in ("split", "routes", "host"):
        cells, es = case["n"] * case["S"], 4 if case["i32"] else 2
        return {"bytes": cells * (es + (2 if op == "routes" else 0)) + 4 * case["S"], "flops": 4 * cells}
    if op == "batch":
        cells = case["T"] * case["S"] * (case["n_lo"] + case["n_hi"]) // 2
        return {"bytes": 2 * cells + 4 * case["T"] * case["S"], "flops": 4 * cells}
    if op == "tours":
        es = 4 if case["i32"] else 2
        return {"bytes": case["n"] * case["S"] * es + 4 * case["T"] * case["n"],
                "flops": 4 * case["T"] * case["n"] * case["S"]}
    if op == "gen":
        cells = case["n"] * case["S"]
        return {"bytes": cells * (4 if case["i32"] else 2), "flops": 60 * cells}
    if op == "search":
        cells = case["k"] * case["n"] * case["S"]
        return {"bytes": case["iterations"] * (2 * case["n"] * case["S"] + 4 * case["M"] * case["n"]),
                "flops": case["iterations"] * (4 * cells + case["M"] * _net_flops(case["n"]))}
    if op == "predict":
        return {"bytes": 4 * case["T"] * (case["n"] + 1), "flops": case["T"] * _net_flops(case["n"])}
    return {"bytes": case["steps"] * (4 * case["T"] * (case["n"] + 1) + 6 * 4 * PARAMS),
            "flops": 3 * case["steps"] * case["T"] * _net_flops(case["n"])}


def _net_flops(n):
    return n * H * (2 * IN1 + 2) + 2 * H * IN2 + 2 * H


# ---------------------------------------------------------------- the same in 64 bits


def _dp(insts, tours, D):
    """Costs (float64 [T][S], inf where infeasible) of tours[t] under D[t] (or one shared matrix), by Eq. 1 over every
    feasible last route."""
    T, S = len(tours), D[0].shape[1]
    n_max = max(len(t) for t in tours)
    dev = D[0].device
    per = max(1, (1 << 30) // (T * n_max))       # scenario columns at once
    out = torch.empty((T, S), dtype=torch.float64, device=dev)
    tab = np.zeros((3, T, n_max + 2), np.int64)  # c(0, s_k), c(s_k, 0), c(s_k, s_k+1)
    for t, (inst, tour) in enumerate(zip(insts, tours)):
        d, n = inst.dist.astype(np.int64), len(tour)
        tab[0, t, 1:n + 1], tab[1, t, 1:n + 1] = d[0, tour], d[tour, 0]
        tab[2, t, 1:n] = d[tour[:-1], tour[1:]]
    length = np.concatenate([np.zeros((T, 1), np.int64), np.cumsum(tab[2][:, 1:], axis=1)], axis=1)  # D[k] at k-1
    tab, length = torch.from_numpy(tab).to(dev), torch.from_numpy(length).to(dev)
    Q = torch.tensor([i.Q for i in insts], device=dev)[:, None]
    L = torch.tensor([min(i.L, i.n) for i in insts], device=dev)[:, None]
    n_of = torch.tensor([len(t) for t in tours], device=dev)
    for a in range(0, S, per):
        b = min(S, a + per)
        P = torch.zeros((n_max + 1, T, b - a), dtype=torch.int64, device=dev)
        for t, tour in enumerate(tours):
            q = D[t if len(D) > 1 else 0][torch.from_numpy(tour.astype(np.int64) - 1).to(dev), a:b].to(torch.int64)
            P[1:len(tour) + 1, t] = q.cumsum(0)
            P[len(tour) + 1:, t] = P[len(tour), t]
        f = torch.full((n_max + 1, T, b - a), math.inf, dtype=torch.float64, device=dev)
        f[0] = 0.0
        for i in range(1, n_max + 1):
            best = f[i]
            for j in range(1, i + 1):
                p = i - j
                ok = (P[i] - P[p] <= Q) & (j <= L)
                if j > 1 and not bool(ok.any()):
                    break
                leg = tab[0, :, p + 1] + (length[:, i - 1] - length[:, p]) + tab[1, :, i]
                cand = f[p] + leg[:, None]
                best = torch.where(ok & (cand < best), cand, best)
            f[i] = best
        out[:, a:b] = f[n_of, torch.arange(T, device=dev)]
    return out


def _saa(cost):
    """(costs with INT32_MAX for infeasible, sum, infeasible, mean) of costs [T][S]."""
    fine = torch.isfinite(cost)
    s = torch.where(fine, cost, 0.0).sum(1)
    k = fine.sum(1)
    return torch.where(fine, cost, float(2**31 - 1)).to(torch.int64), s.to(torch.int64), cost.shape[1] - k, s / k


def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


class Net:
    """The surrogate in 64 bits (weights rounded to BF16, as the network is defined)."""

    def __init__(self, inst, cust, scale, p):
        self.n = inst.n
        c = torch.from_numpy(cust).cuda()
        c = torch.stack([c[:, 0] / 1000.0, c[:, 1] / 1000.0, c[:, 2] / float(inst.Q), c[:, 3] / float(inst.Q)], 1)
        self.c = c.to(torch.float64)
        self.dist = torch.from_numpy(inst.dist).cuda().to(torch.float64)
        self.scale = scale
        self.p = torch.from_numpy(p).cuda().to(torch.float64)

    def parts(self):
        p, o = _bf16(self.p), 0
        got = []
        for shape in ((H, IN1), (H,), (H, IN2), (H,), (H,), (1,)):
            k = math.prod(shape)
            got.append(p[o:o + k].reshape(shape))
            o += k
        return got

    def forward(self, tours):
        w1, b1, w2, b2, w3, b3 = self.parts()
        t = tours.to(torch.int64)
        x = self.c[t - 1]
        cum = x[:, :, 2].cumsum(1)
        phi = torch.cat([x, (cum - cum.floor())[:, :, None]], 2)
        length = self.dist[0, t[:, 0]] + self.dist[t[:, -1], 0] + self.dist[t[:, :-1], t[:, 1:]].sum(1)
        z = []
        for a in range(0, len(t), 256):
            z.append((phi[a:a + 256] @ w1.T + b1).clamp_min(0.0).mean(1))
        zt = torch.cat([torch.cat(z), ((length - self.scale[0]) / self.scale[1])[:, None]], 1)
        u = (zt @ w2.T + b2).clamp_min(0.0)
        return u @ w3 + b3, phi, zt, u

    def step_grad(self, tours, target):
        w1, b1, w2, b2, w3, b3 = self.parts()
        y, phi, zt, u = self.forward(tours)
        T = len(tours)
        e = y - target.to(torch.float64)
        dy = 2.0 * e / T
        du = dy[:, None] * w3 * (u > 0)
        dz = (du @ w2)[:, :H] / self.n
        g1, gb1 = torch.zeros((H, IN1), dtype=torch.float64, device="cuda"), torch.zeros(H, dtype=torch.float64, device="cuda")
        for a in range(0, T, 256):
            d = dz[a:a + 256, None, :] * (phi[a:a + 256] @ w1.T + b1 > 0)
            g1 += d.flatten(0, 1).T @ phi[a:a + 256].flatten(0, 1)
            gb1 += d.sum((0, 1))
        g = torch.cat([g1.ravel(), gb1, (du.T @ zt).ravel(), du.sum(0), dy @ u, dy.sum()[None]])
        return (e ** 2).mean(), g


def exact(case, seed):
    op = case["op"]
    if op in ("gen", "search"):
        return None                              # whole numbers; a path of decisions
    x = _inputs(case, seed)
    if op == "predict":
        inst, cust, tours, scale, target, p, m, v = x
        return {"scores": Net(inst, cust, scale, p).forward(torch.from_numpy(tours).cuda())[0]}
    if op == "train":
        inst, cust, tours, scale, target, p, m, v = x
        net, T, loss = Net(inst, cust, scale, p), case["T"], []
        m, v = (torch.from_numpy(a).cuda().to(torch.float64) for a in (m, v))
        for k in range(case["steps"]):
            at = slice(k * T, (k + 1) * T)
            e, g = net.step_grad(torch.from_numpy(tours[at]).cuda(), torch.from_numpy(target[at]).cuda())
            loss.append(float(e))
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            s = ADAM_STEP + k + 1
            net.p = net.p - LR * (m / (1 - 0.9 ** s)) / ((v / (1 - 0.999 ** s)).sqrt() + 1e-8)
        return {"loss": np.array(loss), "p": net.p, "m": m, "v": v}
    if op == "batch":
        insts, D = x
        costs, s, inf, mean = _saa(_dp(insts, [i.tour for i in insts], D))
        return {"sum": s, "infeasible": inf, "mean": mean, "costs": list(costs[:12])}
    if op == "tours":
        inst, D, tours = x
        _, s, inf, mean = _saa(_dp([inst] * len(tours), list(tours), [D]))
        return {"mean": mean, "sum": s, "infeasible": inf}
    inst, D = x
    costs, s, inf, mean = _saa(_dp([inst], [inst.tour], [D]))
    got = {"costs": costs[0], "sum": int(s[0]), "infeasible": int(inf[0]), "mean": float(mean[0])}
    return {**got, "pred": None} if op == "routes" else got
