"""Parents with objectives that are not finite (nsga3_set_population takes any
values).  One that a generation has to normalise ends it with ENONFINITE and
leaves population and counter as they were; the context then works on."""
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


def _start(n, r):
    r.check(n.nsga3_init(r.ctx, None))
    r.check(n.nsga3_run(r.ctx, 2, None))
    assert r.sync() == 0
    return r.population()


# one warp's solve (m up to 32) and the cluster's; timed phases keep the first
# two off the one-cluster path
REFUSED = [(3, 8, 100, 12, {"phase_timing": 2}), (10, 14, 130, 3, {"phase_timing": 2}),
           (10, 14, 130, 3, {"phase_timing": 2, "norm_history": 1}), (5, 9, 1100, 4, {}), (12, 20, 80, 1, {}),
           (40, 45, 70, 1, {}), (40, 45, 70, 1, {"norm_history": 1})]


@pytest.mark.parametrize("m,d,N,p1,opts", REFUSED)
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_member_to_normalise_is_refused(n, m, d, N, p1, opts, bad):
    with Run(n, m, d, N, p1, seed=3, W=wl.objective_weights(m, 1), **opts) as r:
        X, F, rank = _start(n, r)
        G = F.copy()
        G[N // 2] = -1.0  # below every child elsewhere: in the first front
        G[N // 2, 0] = bad
        r.set_population(X, G, rank)
        for _ in range(2):
            r.check(n.nsga3_step(r.ctx, None))
            assert r.sync() == n.ENONFINITE
            for a, b in zip(r.population(), (X, G, rank)):
                assert np.array_equal(a, b, equal_nan=a.dtype == np.float32)
            assert r.counter() == 2
        r.set_population(X, F, rank)
        r.check(n.nsga3_step(r.ctx, None))
        assert r.sync() == 0 and r.counter() == 3
        assert np.isfinite(r.population()[1]).all()


def _parents(kind, N, m, F):
    """Objectives of N parents, N - 3 of them the given finite ones."""
    G = F.copy()
    if kind == "above":  # three equal rows that every finite one dominates
        G[[1, 4, N - 1]] = np.inf
    else:  # parents below every child and none of them dominated, so that no niching is needed ...
        G = wl.objectives("simplex", N, m, seed=7) - np.float32(5.0)
        G[[1, N - 1]] = -20.0  # ... two equal ones with an infinity
        G[[1, N - 1], 1] = np.inf
        if kind == "minus":
            G[[1, N - 1]] = -3.0
            G[[1, N - 1], 0] = -np.inf
    return G


# (one cluster: odd and even words per CTA, also with the variation outside)
SAME = [(3, 8, 100, 12, {}, {"phase_timing": 2}), (3, 8, 100, 12, {"full_sort": 1}, {"full_sort": 1, "phase_timing": 2}),
        (10, 14, 130, 3, {"full_sort": 1}, {"full_sort": 1, "phase_timing": 2}),
        (7, 40, 1000, 3, {}, {"phase_timing": 2}),
        # the first front before the matrix, and the matrix of all points
        (6, 8, 32768, 3, {}, {"full_sort": 1}), (6, 8, 32790, 3, {"streaming": 1}, {"full_sort": 1})]


@pytest.mark.parametrize("m,d,N,p1,opts,general", SAME)
@pytest.mark.parametrize("kind", ["above", "plus", "minus"])
def test_infinities_compare_as_values(n, m, d, N, p1, opts, general, kind):
    """Equal infinities do not make one row dominate another, or itself: the
    paths with the one-sided pair test against those with the two-sided one."""
    W = wl.objective_weights(m, 1)
    with Run(n, m, d, N, p1, seed=3, W=W, **opts) as a, Run(n, m, d, N, p1, seed=3, W=W, **general) as b:
        out = []
        for r in (a, b):
            X, F, rank = _start(n, r)
            G = _parents(kind, N, m, F)
            r.set_population(X, G, rank)
            r.check(n.nsga3_step(r.ctx, None))
            assert r.sync() == 0
            out.append(r.population() + r.children())
            if kind == "above":
                assert np.isfinite(out[-1][1]).all()
            else:  # the parents stay, all of them in the first front
                assert np.array_equal(out[-1][1], G) and (out[-1][2] == 0).all()
        for x, y in zip(*out):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("m,d,N,p1,opts", [(3, 8, 100, 12, {}), (10, 14, 130, 3, {"norm_history": 1}), (4, 300, 600, 9, {}),
                                           (6, 8, 32768, 3, {})])
def test_member_to_normalise_is_refused_by_the_other_paths(n, m, d, N, p1, opts, bad):
    test_member_to_normalise_is_refused(n, m, d, N, p1, opts, bad)
