"""Timed cases of the NSGA-III library: what its users call, at the sizes they call it.

Three kinds of call, all through the C ABI binding with device buffers:

  select  nsga3_select on a merged 2N x m objective matrix (programs that
          evaluate their own objectives): ranks and selected indices;
  vary    nsga3_vary: the children of one population and their objectives;
  run     nsga3_init + nsga3_run + nsga3_get_population: a whole run from its
          seed; with "runs" > 1 the uneven runs of a batched set advanced
          together by nsga3_run_batch.

A case says the sizes and the options; the seed draws the inputs (objective
matrices, populations, weights of the objective, the Philox key).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2504_06067_gb300 import native as n
from paper_2504_06067_gb300 import workloads as wl


def listed():
    S = dict(kind="select", full_sort=False, streaming=False, norm_history=False)
    R = dict(kind="run", runs=1, problem="simplex", norm_history=False)
    return [
        # the smallest configuration (92 individuals, 91 directions): a
        # program whose own objective is cheap waits for the launches
        dict(S, name="select_m3_N92", m=3, N=92, p1=12, p2=0, shape="early"),
        # the scale configuration, directions about as many as individuals,
        # late in a run (one large front)
        dict(S, name="select_m5_N10628", m=5, N=10628, p1=20, p2=0, shape="late"),
        # the largest eight-objective run of the batched set: association
        # with 11,440 directions
        dict(S, name="select_m8_N19364", m=8, N=19364, p1=9, p2=0, shape="late"),
        # the large population with a two-layer direction set, early in a run
        dict(S, name="select_m10_N100000", m=10, N=100000, p1=3, p2=2, shape="early"),
        # a population whose dominance matrix the caller does not want in memory
        dict(S, name="select_m6_N60000_streaming", m=6, N=60000, p1=6, p2=0, shape="late", streaming=True),
        # variation and objective alone, for programs with their own selection
        dict(kind="vary", name="vary_m5_N10628_d100", m=5, N=10628, d=100),
        # whole runs: the small configuration over its 100 generations ...
        dict(R, name="run_m3_N92_d12", m=3, N=92, d=12, p1=12, p2=0, generations=100),
        # ... the scale configuration ...
        dict(R, name="run_m5_N10628_d100", m=5, N=10628, d=100, p1=20, p2=0, generations=60),
        # ... the large population ...
        dict(R, name="run_m10_N100000_d200", m=10, N=100000, d=200, p1=3, p2=2, generations=20),
        # ... many objectives (the objective sweep: N = 800, d = 1000) ...
        dict(R, name="run_m64_N800_d1000", m=64, N=800, d=1000, p1=1, p2=0, generations=20),
        # ... the 0-1 knapsack, whose integer objectives give many fronts ...
        dict(R, name="run_knapsack_m3_N12800_d500", m=3, N=12800, d=500, p1=158, p2=0, generations=20,
             problem="knapsack"),
        # ... and uneven independent runs advanced together
        dict(R, name="batch_16_runs", m=0, N=20000, d=0, p1=0, p2=0, generations=40, runs=16, mix=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Sizes of the served stream and the sweeps: N log-uniform (even), m from
    2 to 10, a smaller share above; directions about as many as individuals
    or a small two-layer set."""
    what = rng.choice(["select", "select", "select", "vary", "run", "run", "run", "batch"])
    if what == "batch":
        return dict(kind="run", problem="simplex", norm_history=False, m=0, N=20000, d=0, p1=0, p2=0,
                    generations=rng.randint(8, 40), runs=rng.randint(3, 15), mix=rng.randint(1, 10000))
    many = rng.random() < 0.15
    m = rng.randint(11, 100) if many else rng.randint(2, 10)
    N = 2 * _log(rng, 25, 1000 if many else 25000)
    if what == "vary":
        return dict(kind="vary", m=m, N=N, d=m - 1 + _log(rng, 4, 200))
    if not many and rng.random() < 0.3:
        p1, p2 = 3, 2
    else:
        p1, p2 = wl.largest_p(m, N), 0
    hist = rng.random() < 0.2
    if what == "select":
        full = N <= 20000 and rng.random() < 0.15
        return dict(kind="select", m=m, N=N, p1=p1, p2=p2, shape=rng.choice(["early", "late"]), full_sort=full,
                    streaming=m <= 10 and rng.random() < 0.15, norm_history=hist)
    gens = max(4, min(60, 200000 // N))
    knap = m <= 5 and rng.random() < 0.5
    return dict(kind="run", runs=1, problem="knapsack" if knap else "simplex", norm_history=hist, m=m, N=N,
                d=_log(rng, 50, 500) if knap else m - 1 + _log(rng, 4, 200), p1=p1, p2=p2, generations=gens)


# ----------------------------------------------------------------- states ----
class _Contexts:
    """Contexts of one state, destroyed with it."""

    def __init__(self):
        self.ctxs = []

    def create(self, m, d, N, p1, opts):
        ctx = n.create(m, d, N, p1, opts)
        self.ctxs.append(ctx)
        return ctx

    def __del__(self):
        for c in self.ctxs:
            n.nsga3_destroy(c)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _objectives(shape, n2, m, seed):
    """Merged objectives near the unit simplex, the front of the softmax-simplex
    problem: a wide spread of the distance factor early in a run (many fronts),
    a narrow one late (one or two large fronts)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    e = torch.empty(n2, m, device="cuda").exponential_(generator=g)
    e = e / e.sum(dim=1, keepdim=True)
    t = torch.empty(n2, 2, device="cuda").exponential_(generator=g)
    dist = 1.0 + (2.0 * t.sum(dim=1) if shape == "early" else 0.01 * t[:, 0])
    return (e * dist[:, None]).contiguous()


def _population(case, seed):
    """X in [0, 1], objectives near the front, front indices 0..2."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand(case["N"], case["d"], device="cuda", generator=g)
    rank = torch.randint(0, 3, (case["N"],), device="cuda", generator=g, dtype=torch.int32)
    return X, _objectives("late", case["N"], case["m"], seed + 1), rank


def _run_members(case):
    """(m, d, N, p1, p2) of every run of a run case."""
    if case["runs"] == 1:
        return [(case["m"], case["d"], case["N"], case["p1"], case["p2"])]
    return [(c.m, c.d, c.N, c.p1, c.p2) for c in wl.batched_configs(case["runs"], seed=case["mix"])]


def prepare(case, seed):
    st = {"case": case, "own": _Contexts()}
    own = st["own"]
    if case["kind"] == "select":
        o = n.default_opts(seed=seed, p2=case["p2"], full_sort=int(case["full_sort"]),
                           streaming=int(case["streaming"]), norm_history=int(case["norm_history"]))
        st["ctx"] = own.create(case["m"], max(1, case["m"] - 1), case["N"], case["p1"], o)
        st["objs"] = _objectives(case["shape"], 2 * case["N"], case["m"], seed)
        st["ranks"] = torch.empty(2 * case["N"], dtype=torch.int32, device="cuda")
        st["selected"] = torch.empty(case["N"], dtype=torch.int32, device="cuda")
        n.check(n.nsga3_set_counter(st["ctx"], seed % 1000, _stream()), st["ctx"])
        return st
    if case["kind"] == "vary":
        W = wl.objective_weights(case["m"], seed)
        ctx = st["ctx"] = own.create(case["m"], case["d"], case["N"], 1, n.default_opts(seed=seed, W=W.ctypes.data))
        X, F, rank = _population(case, seed)
        s = _stream()
        n.check(n.nsga3_set_population(ctx, X.data_ptr(), F.data_ptr(), rank.data_ptr(), s), ctx)
        n.check(n.nsga3_set_counter(ctx, seed % 1000, s), ctx)
        n.check(n.nsga3_sync(ctx, s), ctx)  # X, F and rank are copied
        st["X"], st["F"] = torch.empty_like(X), torch.empty_like(F)
        return st
    st["ctxs"], st["out"] = [], []
    for r, (m, d, N, p1, p2) in enumerate(_run_members(case)):
        key = dict(seed=seed * 64 + r, p2=p2, norm_history=int(case["norm_history"]))
        if case["problem"] == "knapsack":
            kp = wl.knapsack_instance(m, d, seed)
            key.update(problem=1, kp_profit=kp[0].ctypes.data, kp_weight=kp[1].ctypes.data,
                       kp_capacity=kp[2].ctypes.data)
        else:
            W = wl.objective_weights(m, seed * 64 + r)
            key.update(W=W.ctypes.data)
        st["ctxs"].append(own.create(m, d, N, p1, n.default_opts(**key)))
        st["out"].append((torch.empty(N, d, device="cuda"), torch.empty(N, m, device="cuda"),
                          torch.empty(N, dtype=torch.int32, device="cuda")))
    return st


def run(st):
    case, s = st["case"], _stream()
    if case["kind"] == "select":
        ctx = st["ctx"]
        n.check(n.nsga3_select(ctx, st["objs"].data_ptr(), st["ranks"].data_ptr(), st["selected"].data_ptr(), s), ctx)
        return {"ranks": st["ranks"], "selected": st["selected"]}
    if case["kind"] == "vary":
        ctx = st["ctx"]
        n.check(n.nsga3_vary(ctx, s), ctx)
        n.check(n.nsga3_get_children(ctx, st["X"].data_ptr(), st["F"].data_ptr(), s), ctx)
        return {"X": st["X"], "F": st["F"]}
    ctxs = st["ctxs"]
    for ctx in ctxs:
        n.check(n.nsga3_init(ctx, s), ctx)
    if len(ctxs) == 1:
        n.check(n.nsga3_run(ctxs[0], case["generations"], s), ctxs[0])
    else:
        n.check(n.run_batch(ctxs, case["generations"], s), ctxs[0])
    for ctx, (X, F, rank) in zip(ctxs, st["out"]):
        n.check(n.nsga3_get_population(ctx, X.data_ptr(), F.data_ptr(), rank.data_ptr(), s), ctx)
    return [list(o) for o in st["out"]]


# ------------------------------------------------------------------- work ----
def work(case):
    """Bytes: inputs read once and outputs written once (for a run, each
    generation's parents, children and merged objectives).  Operations: the
    arithmetic of the objective and of one distance per associated point;
    the dominance tests and the search for the nearest direction can be
    pruned and are not counted."""
    if case["kind"] == "select":
        n2, m = 2 * case["N"], case["m"]
        return {"bytes": 4.0 * (n2 * m + n2 + case["N"]), "flops": 4.0 * n2 * m}
    if case["kind"] == "vary":
        N, m, d = case["N"], case["m"], case["d"]
        return {"bytes": 4.0 * N * (2 * d + m + 1), "flops": N * (8.0 * d + 2.0 * m * (m - 1))}
    b = f = 0.0
    for m, d, N, _, _ in _run_members(case):
        # a generation: parents read, children written, merged objectives read
        b += case["generations"] * 4.0 * N * (2 * d + 3 * m + 2) + 4.0 * N * (d + m + 1)
        f += case["generations"] * N * (8.0 * d + 2.0 * m * (m - 1) + 8.0 * m)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact ----
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 on int64 tensors (c0; the other words are numbers)."""
    c = [c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.full_like(c0, c3)]
    k0, k1 = key & _M32, (key >> 32) & _M32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # 64-bit products, modulo 2^64
        c = [((b >> 32) & _M32) ^ c[1] ^ k0, b & _M32, ((a >> 32) & _M32) ^ c[3] ^ k1, a & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _u01(w):
    return (w >> 8).double() * 2.0 ** -24


def _mutate(y, u, eta):
    low = u < 0.5
    pw = torch.where(low, 1.0 - y, y) ** (eta + 1.0)
    val = torch.where(low, 2.0 * u + (1.0 - 2.0 * u) * pw, 2.0 * (1.0 - u) + 2.0 * (u - 0.5) * pw)
    dq = torch.expm1(torch.log(val) / (eta + 1.0))
    return (y + torch.where(low, dq, -dq)).clamp(0.0, 1.0)


def exact(case, seed):
    """Variation: simulated binary crossover, polynomial mutation and the
    objective in 64 bits.  Selections return whole numbers, and a run's
    selections turn on its roundings: no value."""
    if case["kind"] != "vary":
        return None
    N, m, d, gen = case["N"], case["m"], case["d"], seed % 1000
    X, _, rank = _population(case, seed)
    X = X.double()
    q = torch.arange(N // 2, device="cuda", dtype=torch.int64)
    t = _philox(q, gen, 1, 0, seed)
    a = [(w * N) >> 32 for w in t]
    pick = [torch.where(rank[a[k + 1]] < rank[a[k]], a[k + 1], a[k]) for k in (0, 2)]
    y1, y2 = X[pick[0]], X[pick[1]]
    cross = _u01(_philox(q, gen, 1, 1, seed)[0]) < 1.0
    qv = (q[:, None] * d + torch.arange(d, device="cuda")) & _M32
    sb = _philox(qv, gen, 2, 0, seed)
    u = _u01(sb[0])
    beta = torch.where(u <= 0.5, 2.0 * u, 1.0 / (2.0 * (1.0 - u))) ** (1.0 / 21.0)
    c1 = 0.5 * ((1.0 + beta) * y1 + (1.0 - beta) * y2)
    c2 = 0.5 * ((1.0 - beta) * y1 + (1.0 + beta) * y2)
    swap = _u01(sb[2]) < 0.5
    c1, c2 = torch.where(swap, c2, c1).clamp(0.0, 1.0), torch.where(swap, c1, c2).clamp(0.0, 1.0)
    do = cross[:, None] & (_u01(sb[1]) < 0.5)
    c1, c2 = torch.where(do, c1, y1), torch.where(do, c2, y2)
    pm, p_m = _philox(qv, gen, 3, 0, seed), float(np.float32(1.0) / np.float32(d))
    c1 = torch.where(_u01(sb[3]) < p_m, _mutate(c1, _u01(pm[0]), 20.0), c1)
    c2 = torch.where(_u01(pm[1]) < p_m, _mutate(c2, _u01(pm[2]), 20.0), c2)
    C = torch.stack([c1, c2], dim=1).reshape(N, d)
    W = torch.from_numpy(wl.objective_weights(m, seed)).double().cuda()
    g = ((C[:, m - 1:] - 0.5) ** 2).sum(dim=1, keepdim=True)
    F = (1.0 + g) * torch.softmax(C[:, :m - 1] @ W.T, dim=1)
    return {"X": C, "F": F}
