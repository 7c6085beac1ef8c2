"""The first front before the matrix (large populations, m >= 5) against the
path without it: a complete ranking (full_sort = 1) builds the matrix of all
points.  The fronts up to F_l, the selected indices and the normalization
agree, with a rest (many fronts) and without one (the first front holds N),
at the smallest size that takes the path, whole and ragged blocks of 32, with
and without the matrix in memory."""
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


@pytest.mark.parametrize("shape", [(5, 39322, 0), (6, 32768, 1), (7, 32782, 0), (8, 32800, 0), (9, 33000, 1),
                                   (10, 32770, 0)])
def test_first_front_matches_the_whole_matrix(n, shape):
    m, N, streaming = shape
    with Run(n, m, m + 1, N, 3, seed=5, streaming=streaming) as a, Run(n, m, m + 1, N, 3, seed=5, full_sort=1) as b:
        for kind in ("early", "late", "uniform", "equal", "dups", "grid", "signedzero"):
            F = wl.objectives(kind, 2 * N, m, seed=3)
            st, rank, sel = a.select(F, gen=2)
            st2, rank2, sel2 = b.select(F, gen=2)
            assert st == 0 and st2 == 0, kind
            ia, ib = a.info(), b.info()
            for k in ("l", "nS", "K", "nFl"):
                assert ia[k] == ib[k], (kind, k)
            assert np.array_equal(rank, np.where(rank2 <= ib["l"], rank2, -1)), kind
            assert np.array_equal(sel, sel2), kind
            for x, y in zip(a.normalization(), b.normalization()):
                assert np.array_equal(x, y), kind


def test_first_front_then_few_points_left(n):
    """Rests of no, one and a few points short of N, and of one tile and one
    point more: a first front of N - k points on a simplex above a cloud that
    it dominates."""
    m, N = 6, 32768
    with Run(n, m, m + 1, N, 3, seed=5) as a, Run(n, m, m + 1, N, 3, seed=5, full_sort=1) as b:
        for first in (N, N - 1, N + 1, 2 * N - 1, 2 * N - 256, 2 * N - 257, 1):
            F = wl.objectives("simplex", 2 * N, m, seed=first)
            rng = np.random.default_rng(first)
            order = rng.permutation(2 * N)
            F[order[first:]] = F[order[rng.integers(0, first, 2 * N - first)]] + np.float32(0.125)
            st, rank, sel = a.select(F, gen=1)
            st2, rank2, sel2 = b.select(F, gen=1)
            assert st == 0 and st2 == 0
            l = b.info()["l"]
            assert a.info()["l"] == l
            assert np.array_equal(rank, np.where(rank2 <= l, rank2, -1)), first
            assert np.array_equal(sel, sel2), first
