"""Niche selection of the one-cluster path where few directions share many
members: lists around the length from which all of F_l is sorted, whole
populations at one direction, equal distances, with and without members of
earlier fronts (rho), against the oracle."""
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


def _near_axes(counts, m, rng):
    """counts[q] points of the unit simplex near axis q."""
    rows = []
    for q, k in enumerate(counts):
        U = rng.dirichlet(np.ones(m), size=k)
        rows.append(0.9 * np.eye(m)[q] + 0.1 * U)
    return np.vstack(rows)


def _check(n, orc, r, F, Z):
    k = C.c_int32()
    for gen in (0, 5):
        st, rank, sel = r.select(F, gen=gen)
        assert st == 0
        r.check(n.nsga3_last_launches(r.ctx, C.byref(k)))
        assert k.value == 1
        ref = orc.select(F, r.N, Z, seed=9, gen=gen)
        assert ref["niche"]
        assert np.array_equal(rank, ref["rank"]) and np.array_equal(sel, ref["selected"])


@pytest.mark.parametrize("early", [0, 5])
@pytest.mark.parametrize("counts", [(31, 1, 4), (32, 3, 2), (33, 2, 2), (34, 33, 32), (65, 0, 1), (400, 333, 33), (1024, 3, 1),
                                    (1500, 300, 200), (256, 250, 3), (257, 250, 2), (128, 500, 0), (129, 480, 300),
                                    (85, 900, 20), (86, 900, 80), (64, 1000, 800), (65, 65, 1900)])
def test_lists_of_one_direction(n, orc, counts, early):
    """`early` members of an earlier front near each axis: rho > 0."""
    m, rng = 3, np.random.default_rng(sum(counts) + early)
    U = _near_axes(counts, m, rng)
    if early:
        U = np.vstack([0.98 * _near_axes((early,) * m, m, rng), U + 0.12])
    k = len(U)
    N = (k + 3) // 4 * 2
    if early:
        N = max(N, 2 * ((3 * early + 3) // 2))
    F = np.vstack([U, U[rng.integers(0, k, 2 * N - k)] + 2.0]) if 2 * N > k else U
    F = F[rng.permutation(2 * N)].astype(np.float32)
    Z = orc.refdirs(m, 1)
    with Run(n, m, m, N, 1, seed=9) as r:
        _check(n, orc, r, F, Z)


@pytest.mark.parametrize("m,N,p1", [(2, 1024, 1), (2, 18, 1), (5, 1000, 2), (10, 1024, 1), (3, 514, 1)])
@pytest.mark.parametrize("kind", ["equal", "late", "grid", "simplex", "dups"])
def test_few_directions(n, orc, m, N, p1, kind):
    Z = orc.refdirs(m, p1)
    F = wl.objectives(kind, 2 * N, m, seed=2)
    if not orc.select(F, N, Z, seed=9, gen=0)["niche"]:
        pytest.skip("no niching")
    with Run(n, m, m, N, p1, seed=9) as r:
        _check(n, orc, r, F, Z)
