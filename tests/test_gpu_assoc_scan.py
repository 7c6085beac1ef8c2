"""The association's tensor-core scan (m <= 10, general path) against the oracle
where it can go wrong: directions and points around whole blocks of 32,
chunks of 128 and groups of 256, more chunks than the ring holds and several
items per CTA, points on axes, at the centre and between directions, and the
scale configuration.  The FP64 scan of every direction (debug_recheck_all)
must agree for every m."""
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


def _check(orc, r, F, Z, gen):
    st, rank, sel = r.select(F, gen=gen)
    assert st == 0
    ref = orc.select(F, r.N, Z, seed=4, gen=gen)
    assert ref["niche"]
    assert np.array_equal(rank, ref["rank"])
    pi, dist = r.association()
    T = (ref["rank"] >= 0) & (ref["rank"] <= ref["l"])
    assert np.array_equal(pi[T], ref["pi"][T]) and np.array_equal(dist[T], ref["dist"][T])
    assert np.array_equal(sel, ref["selected"])
    return r.info()


def _first(U, n2, seed):
    """A first front of the points U (on the unit simplex) among n2 points, in
    random order: the others are dominated."""
    rng = np.random.default_rng(seed)
    F = np.vstack([U, U[rng.integers(0, len(U), n2 - len(U))] + 0.5])
    return F[rng.permutation(n2)].astype(np.float32)


def _simplex(k, m, seed):
    return np.random.default_rng([seed, m]).dirichlet(np.ones(m), size=k)


@pytest.mark.parametrize("w", [2, 3, 31, 32, 33, 127, 128, 129, 255, 256, 257, 1025, 3000])
def test_directions_around_blocks_and_chunks(n, orc, w):
    """m = 2 takes any number of directions; the smallest is two."""
    N = 200
    Z = orc.refdirs(2, w - 1)
    assert len(Z) == w
    with Run(n, 2, 2, N, w - 1, seed=4, phase_timing=2) as r:
        _check(orc, r, _first(_simplex(300, 2, w), 2 * N, w), Z, 3)


@pytest.mark.parametrize("k", [127, 128, 129, 255, 256, 257, 383, 384, 385, 511, 512, 513])
def test_points_around_groups(n, orc, k):
    m, p1 = 4, 9
    N = 2 * ((k + 3) // 4)
    Z = orc.refdirs(m, p1)
    with Run(n, m, m, N, p1, seed=4, phase_timing=2) as r:
        info = _check(orc, r, _first(_simplex(k, m, k), 2 * N, k), Z, 1)
        assert info["nT"] == k


# chunks per item beyond the ring of eight, several items per CTA; FP16 rows of
# 16 halves (m <= 5) and of 32
@pytest.mark.parametrize("m,N,p1", [(3, 3000, 100), (5, 6000, 13), (6, 4000, 9), (8, 2500, 8)])
def test_many_chunks_and_items(n, orc, m, N, p1):
    Z = orc.refdirs(m, p1)
    with Run(n, m, m, N, p1, seed=4, phase_timing=2) as r:
        _check(orc, r, _first(_simplex(2 * N - 7, m, 5), 2 * N, 5), Z, 2)


@pytest.mark.parametrize("m", range(2, 11))
def test_every_direction_agrees(n, orc, m):
    """Points at random, within 1e-7 .. 1e-2 of an axis, of the centre, of the
    middle between two directions and of a direction."""
    rng = np.random.default_rng(m)
    p1 = {2: 700, 3: 36, 4: 14, 5: 9, 6: 7, 7: 6, 8: 5, 9: 5, 10: 4}[m]
    Z = orc.refdirs(m, p1)
    k = 1200
    U = _simplex(k, m, 1)
    i, j = rng.integers(0, len(Z), (2, k))
    at = [np.eye(m)[rng.integers(0, m, k)], np.full((k, m), 1.0 / m), 0.5 * (Z[i] + Z[j]), Z[i]]
    for g, c in enumerate(at):
        sl = slice(200 * (g + 1), 200 * (g + 2))
        eps = 10.0 ** rng.uniform(-7, -2, (200, 1))
        U[sl] = (1.0 - eps) * c[sl] + eps * U[sl]
    N = 2 * (k // 4 + 10)
    F = _first(U, 2 * N, m)
    with Run(n, m, m, N, p1, seed=4, phase_timing=2) as r, \
            Run(n, m, m, N, p1, seed=4, debug_recheck_all=1) as a:
        _check(orc, r, F, Z, 2)
        assert _check(orc, a, F, Z, 2)["recheck_miss"] == 0


def test_no_variable_chooses_the_path(n, monkeypatch):
    import ctypes as C
    k = C.c_int32()
    monkeypatch.setenv("NSGA3_ASSOC", "tile")
    with Run(n, 3, 3, 92, 12, seed=4) as r:
        r.select(wl.objectives("late", 184, 3, seed=1))
        r.check(n.nsga3_last_launches(r.ctx, C.byref(k)))
        assert k.value == 1  # the one cluster of small populations


def test_limit_of_directions(n):
    """m = 2: 126,368 directions are taken, one more is refused."""
    most = (220 * 1024 - 4096) // ((4 + 10) * 4) * 32
    with Run(n, 2, 2, 100, most - 1, seed=1, phase_timing=2) as r:
        assert r.w == most
        st, rank, sel = r.select(wl.objectives("late", 200, 2, seed=1))
        assert st == 0
    with pytest.raises(Exception):
        Run(n, 2, 2, 100, most, seed=1, phase_timing=2)


# many points that tie with directions of many blocks: objectives of a few
# values, with few directions and many
@pytest.mark.parametrize("m,N,p1", [(2, 1500, 300), (3, 2000, 40), (5, 4000, 8), (7, 2000, 4), (10, 5000, 5), (10, 3000, 2)])
@pytest.mark.parametrize("kind", ["dups", "grid", "signedzero"])
def test_many_ties(n, orc, m, N, p1, kind):
    Z = orc.refdirs(m, p1)
    F = wl.objectives(kind, 2 * N, m, seed=4)
    with Run(n, m, m, N, p1, seed=4) as r:
        st, rank, sel = r.select(F, gen=1)
        ref = orc.select(F, N, Z, seed=4, gen=1)
        assert st == 0 and np.array_equal(rank, ref["rank"]) and np.array_equal(sel, ref["selected"])
        if ref["niche"]:
            _check(orc, r, F, Z, 1)


@pytest.mark.parametrize("k", [151, 153, 2000, 2190])
def test_more_ties_than_slots(n, orc, k):
    """k points at the centre, as near to 120 directions, among points near
    directions: whole and ragged groups."""
    m, N, p1 = 10, 1100, 3
    Z = orc.refdirs(m, p1)
    F = _simplex(2 * N, m, 3)
    F[:m] = np.eye(m)
    F[m:m + k] = 1.0 / m
    F = F[np.random.default_rng(k).permutation(2 * N)].astype(np.float32)
    with Run(n, m, m, N, p1, seed=4) as r:
        _check(orc, r, F, Z, 2)


@pytest.mark.parametrize("kind", ["late", "early"])
def test_scale_configuration(n, orc, kind):
    cfg = wl.SCALE
    Z = orc.refdirs(cfg.m, cfg.p1)
    with Run(n, cfg.m, cfg.d, cfg.N, cfg.p1, seed=4) as r:
        _check(orc, r, wl.objectives(kind, 2 * cfg.N, cfg.m, seed=3), Z, 4)
