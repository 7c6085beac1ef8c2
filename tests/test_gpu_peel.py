"""The peel's chunks that are passed over while their counts allow it: one
chunk per CTA, several per CTA, more front words than are kept in shared
memory, with and without the matrix, over many fronts.  Layers with known
ranks (layer t lies below every point of layer t + 1), and random many-front
points against the oracle's complete ranking."""
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


def _layers(n2, m, sizes, seed):
    """Points of len(sizes) layers in random order, and their ranks."""
    rng = np.random.default_rng(seed)
    rank = np.repeat(np.arange(len(sizes)), sizes)[:n2]
    s = rng.dirichlet(np.ones(m), size=n2)
    s = np.round(s * 256) / 256
    s[:, -1] = 2.0 - s[:, :-1].sum(axis=1)  # the same sum exactly: no point of a layer dominates another
    F = (s + 4.0 * rank[:, None]).astype(np.float32)
    order = rng.permutation(n2)
    return F[order], rank[order]


@pytest.mark.parametrize("case", [(3, 1100, 0, {}), (4, 10000, 0, {}), (4, 10000, 0, {"peel_ctas_per_sm": 1}),
                                  (3, 10000, 1, {}), (3, 33000, 0, {}), (12, 1500, 0, {})])
def test_layers_of_known_rank(n, case):
    m, N, streaming, opts = case
    n2 = 2 * N
    for full in (0, 1):
        for sizes in ([n2 // 33 + 1] * 33, [1, 31, 2, n2 // 2, 1, 1, 1, n2], [n2 - 9] + [1] * 9):
            F, want = _layers(n2, m, sizes, seed=len(sizes))
            with Run(n, m, m + 1, N, 2, seed=1, full_sort=full, streaming=streaming, **opts) as r:
                st, rank, sel = r.select(F, gen=3)
            assert st == 0
            l = int(np.sort(want)[N - 1])
            if not full:
                want = np.where(want <= l, want, -1)
            assert np.array_equal(rank, want), (full, sizes[:3])
            assert len(set(sel.tolist())) == N and (rank[sel] <= l).all()


@pytest.mark.parametrize("case", [(3, 600, {}), (2, 2200, {}), (3, 9800, {"peel_ctas_per_sm": 1})])
def test_many_fronts_match_the_oracle(n, orc, case):
    m, N, opts = case
    Z = orc.refdirs(m, 6)
    for kind in ("early", "grid", "uniform"):
        F = wl.objectives(kind, 2 * N, m, seed=4)
        ref = orc.select(F, N, Z, seed=2, gen=1, full_sort=True)
        for streaming in (0, 1):
            with Run(n, m, m + 1, N, 6, seed=2, full_sort=1, streaming=streaming, **opts) as r:
                st, rank, sel = r.select(F, gen=1)
            assert st == 0
            assert np.array_equal(rank, ref["rank"]), (kind, streaming)
            assert np.array_equal(sel, ref["selected"]), (kind, streaming)
