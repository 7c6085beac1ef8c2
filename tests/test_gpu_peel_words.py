"""The peel with several chunks per CTA and more front words than are kept in
shared memory: passes of few front words, whose words are listed, between
passes of many, around the number that is listed.  Layers with known ranks."""
import numpy as np
import pytest

from gpu_util import Run
from test_gpu_peel import _layers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def n():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_2504_06067_gb300 import native
    return native


@pytest.mark.parametrize("m,N,opts", [(3, 33000, {}), (3, 50000, {}), (4, 40000, {"peel_ctas_per_sm": 1}), (10, 33000, {}),
                                      (12, 33000, {})])
def test_sparse_and_dense_passes(n, m, N, opts):
    sizes = [1] * 40 + [900, 1000, 1024, 1056, 1100, 2, 31, 32, 33] + [1] * 7 + [N // 2] + [1] * 8 + [3000] + [40] * 30
    sizes += [2 * N]  # the rest
    F, want = _layers(2 * N, m, sizes, seed=m)
    with Run(n, m, m + 1, N, 1, seed=1, full_sort=1, **opts) as r:
        st, rank, sel = r.select(F, gen=3)
    assert st == 0 and np.array_equal(rank, want)
    l = int(np.sort(want)[N - 1])
    assert len(set(sel.tolist())) == N and (want[sel] <= l).all()
    assert set(np.flatnonzero(want < l)) <= set(sel.tolist())
