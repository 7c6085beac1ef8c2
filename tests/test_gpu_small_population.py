"""Small populations (one launch of one cluster) against the general path over
every form the rule accepts: the same ranks, selections, normalization,
association and next populations, whole numbers and FP64 values bit for bit.
Timed phases (opts.phase_timing) keep a context on the general path."""
import ctypes as C

import numpy as np
import pytest

from paper_2504_06067_gb300 import workloads as wl

from gpu_util import Run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def n():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_2504_06067_gb300 import native
    return native


def _launches(n, r):
    k = C.c_int32()
    r.check(n.nsga3_last_launches(r.ctx, C.byref(k)))
    return k.value


def _same_selection(a, b, F, gen):
    ra, rb = a.select(F, gen), b.select(F, gen)
    assert ra[0] == rb[0]
    assert np.array_equal(ra[1], rb[1])
    if ra[0]:
        return
    assert np.array_equal(ra[2], rb[2])
    ia, ib = a.info(), b.info()
    for k in ("l", "nS", "K", "nFl", "niche", "passes"):
        assert ia[k] == ib[k], k
    if ia["niche"]:
        for k in ("fallback", "nT", "Lstar", "rlev"):
            assert ia[k] == ib[k], k
        for x, y in zip(a.normalization(), b.normalization()):
            assert np.array_equal(x, y)
        inT = (ra[1] >= 0) & (ra[1] <= ia["l"])
        for x, y in zip(a.association(), b.association()):
            assert np.array_equal(x[inT], y[inT])


# merged sizes at the edges of words, CTAs and cluster sizes; directions from
# two to the most the path takes (m = 2, p = 2047)
SIZES = [(3, 2, 1, 0), (2, 16, 5, 0), (3, 32, 6, 2), (4, 34, 3, 0), (5, 64, 3, 2), (3, 92, 12, 0), (6, 130, 3, 0),
         (10, 162, 2, 1), (7, 256, 3, 0), (2, 300, 2047, 0), (8, 512, 5, 0), (9, 514, 3, 2), (10, 800, 3, 0),
         (5, 1022, 11, 0), (3, 1024, 40, 0)]


@pytest.mark.parametrize("m,N,p1,p2", SIZES)
def test_selections_equal_the_general_path(n, m, N, p1, p2):
    with Run(n, m, m + 1, N, p1, p2=p2, seed=7) as a, \
            Run(n, m, m + 1, N, p1, p2=p2, seed=7, phase_timing=2) as b:
        for s, kind in enumerate(wl.KINDS):
            if kind == "chain" and N > 200:
                continue
            _same_selection(a, b, wl.objectives(kind, 2 * N, m, seed=s), 3 + s)
        assert _launches(n, a) == 1 and _launches(n, b) > 1


@pytest.mark.parametrize("opt", ["full_sort", "norm_history", "streaming"])
@pytest.mark.parametrize("m,N,p1", [(3, 100, 8), (10, 210, 3)])
def test_options_equal_the_general_path(n, opt, m, N, p1):
    with Run(n, m, m + 1, N, p1, seed=2, **{opt: 1}) as a, \
            Run(n, m, m + 1, N, p1, seed=2, phase_timing=2, **{opt: 1}) as b:
        for s, kind in enumerate(("early", "late", "grid", "late", "equal", "early")):
            _same_selection(a, b, wl.objectives(kind, 2 * N, m, seed=20 + s), s)


@pytest.mark.parametrize("m,d,N,p1,opts", [
    (3, 12, 92, 12, {}), (5, 24, 200, 6, {}), (2, 1, 64, 30, {}), (10, 40, 100, 2, {"norm_history": 1}),
    (4, 300, 600, 9, {}), (8, 27, 1000, 4, {})])  # the last three vary in a launch of their own
def test_runs_equal_the_general_path(n, m, d, N, p1, opts):
    W = wl.objective_weights(m, 4)
    with Run(n, m, d, N, p1, seed=11, W=W, **opts) as a, \
            Run(n, m, d, N, p1, seed=11, W=W, phase_timing=2, **opts) as b:
        for r in (a, b):
            r.check(n.nsga3_init(r.ctx, None))
            r.check(n.nsga3_run(r.ctx, 25, None))
            assert r.sync() == 0 and r.counter() == 25
        for x, y in zip(a.population() + a.children(), b.population() + b.children()):
            assert np.array_equal(x, y)


def test_knapsack_run_equals_the_general_path(n):
    m, d, N = 3, 50, 150
    p, w, c = wl.knapsack_instance(m, d, 1)
    kp = dict(problem=1, kp_profit=p.ctypes.data, kp_weight=w.ctypes.data, kp_capacity=c.ctypes.data)
    with Run(n, m, d, N, 14, seed=3, **kp) as a, Run(n, m, d, N, 14, seed=3, phase_timing=2, **kp) as b:
        for r in (a, b):
            r.check(n.nsga3_init(r.ctx, None))
            r.check(n.nsga3_run(r.ctx, 15, None))
        for x, y in zip(a.population(), b.population()):
            assert np.array_equal(x, y)


def test_more_near_equal_directions_than_slots(n):
    """Ten directions at the same distance of every member: the FP64 scan of
    all directions decides (the first direction wins)."""
    m, N = 10, 320
    F = np.full((2 * N, m), 0.09, np.float32)
    F[:m] = np.eye(m, dtype=np.float32)
    with Run(n, m, m, N, 1, seed=1) as a, Run(n, m, m, N, 1, seed=1, phase_timing=2) as b:
        _same_selection(a, b, F, 2)
        assert a.info()["overflow"] > 0


def test_device_buffers_and_non_finite_objectives(n):
    import torch
    m, N = 4, 75 * 2
    F = wl.objectives("early", 2 * N, m, seed=5)
    with Run(n, m, m, N, 6, seed=9) as a:
        st, rank, sel = a.select(F, 1)
        Fd = torch.from_numpy(np.concatenate([[0.0], F.ravel()]).astype(np.float32)).cuda()[1:]  # off 16 bytes
        rd = torch.full((2 * N + 1,), 7, dtype=torch.int32, device="cuda")
        sd = torch.full((N + 1,), 7, dtype=torch.int32, device="cuda")
        a.check(n.nsga3_select(a.ctx, Fd.data_ptr(), rd.data_ptr(), sd.data_ptr(), None))
        assert a.sync() == 0
        assert np.array_equal(rd.cpu().numpy()[:-1], rank) and np.array_equal(sd.cpu().numpy()[:-1], sel)
        assert int(rd[-1]) == 7 and int(sd[-1]) == 7
        for bad in (np.nan, np.inf, -np.inf):
            G = F.copy()
            G[-1, -1] = bad
            st, rank_bad, _ = a.select(G, 1)
            assert st == n.ENONFINITE and np.all(rank_bad == -1)
        st, again, sel2 = a.select(F, 1)
        assert st == 0 and np.array_equal(again, rank) and np.array_equal(sel2, sel)
