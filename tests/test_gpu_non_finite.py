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
