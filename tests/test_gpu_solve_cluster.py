"""The intercept system of more than 32 objectives, solved in the shared memory of
one cluster: every group size of its threads (m just below and above a
multiple of 32), both cluster sizes, regular
systems and singular ones (the nadir fallback).  Intercepts bit for bit against
the oracle."""
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


def _corners(n2, m, seed):
    """Points near the simplex and one near each vertex, in random order."""
    rng = np.random.default_rng([seed, m])
    F = rng.dirichlet(np.ones(m), size=n2) * (1.0 + rng.exponential(0.05, size=(n2, 1)))
    k = min(m, n2)
    C = 0.02 * rng.random((k, m)) / m
    C[np.arange(k), np.arange(k)] = 0.9 + 0.05 * rng.random(k)
    F[rng.permutation(n2)[:k]] = C
    return F.astype(np.float32)


@pytest.mark.parametrize("m", [33, 64, 65, 96, 97, 128, 129, 160, 224, 255, 256, 257, 400])
def test_intercepts_match_the_oracle(n, orc, m):
    N = 2 * ((m + 40) // 2)
    Z = orc.refdirs(m, 1)
    with Run(n, m, m + 1, N, 1, seed=3) as r:
        for kind in ("corners", "late", "equal", "grid"):
            F = _corners(2 * N, m, 1) if kind == "corners" else wl.objectives(kind, 2 * N, m, seed=2)
            st, rank, sel = r.select(F, gen=4)
            assert st == 0
            ref = orc.select(F, N, Z, seed=3, gen=4)
            assert np.array_equal(rank, ref["rank"]), kind
            if ref["niche"]:
                z, a, e = r.normalization()
                zs, aa, ee, fb = orc.normalize(F, ref["rank"], ref["l"])
                assert np.array_equal(z, zs) and np.array_equal(e, ee), kind
                assert np.array_equal(a, aa), kind
                assert bool(r.info()["fallback"]) == fb, kind
                if kind == "corners":
                    assert not fb  # the elimination ran to its end
            assert np.array_equal(sel, ref["selected"]), kind
