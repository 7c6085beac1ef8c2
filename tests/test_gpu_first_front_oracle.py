"""The first front before the matrix against the oracle, at the smallest sizes
that take the path: ranks, selected indices and the association."""
import numpy as np
import pytest

from paper_2504_06067_gb300 import workloads as wl

from gpu_util import Run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,N,p1,streaming,kind", [(6, 32768, 4, 0, "early"), (6, 32768, 4, 0, "grid"),
                                                    (10, 32770, 2, 1, "early")])
def test_first_front_matches_the_oracle(orc, m, N, p1, streaming, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_2504_06067_gb300 import native as n
    F = wl.objectives(kind, 2 * N, m, seed=6)
    ref = orc.select(F, N, orc.refdirs(m, p1), seed=5, gen=3)
    with Run(n, m, m, N, p1, seed=5, streaming=streaming) as r:
        st, rank, sel = r.select(F, gen=3)
        assert st == 0
        assert np.array_equal(rank, ref["rank"]) and np.array_equal(sel, ref["selected"])
        if ref["niche"]:
            pi, dist = r.association()
            T = (ref["rank"] >= 0) & (ref["rank"] <= ref["l"])
            assert np.array_equal(pi[T], ref["pi"][T]) and np.array_equal(dist[T], ref["dist"][T])
