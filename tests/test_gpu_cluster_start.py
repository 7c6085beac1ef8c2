"""Small populations while other work holds the SMs: the CTAs of the one cluster
start at different times, and none may store into the shared memory of one
that has not started (a cluster barrier precedes the first such store in
every mode).  Selections, and generations whose variation is a launch of its
own, at every cluster size, equal the oracle's and the undisturbed ones."""
import numpy as np
import pytest

from paper_2504_06067_gb300 import workloads as wl

from gpu_util import Run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    return torch


def _busy(torch, stream, x):
    with torch.cuda.stream(stream):
        for _ in range(4):
            torch.sin(x, out=x)


# 2N at most 32, 64, 128, 512 and 2,048: clusters of 1, 2, 4, 8 and 16 CTAs
@pytest.mark.parametrize("m,N,p1", [(3, 16, 4), (2, 30, 9), (5, 64, 3), (3, 92, 12), (10, 600, 3)])
def test_selections_beside_other_work(torch, orc, m, N, p1):
    from paper_2504_06067_gb300 import native as n
    x = torch.rand(1 << 24, device="cuda")
    side = torch.cuda.Stream()
    Z = orc.refdirs(m, p1)
    with Run(n, m, m, N, p1, seed=6) as r:
        for kind in ("early", "late"):
            F = wl.objectives(kind, 2 * N, m, seed=N)
            ref = orc.select(F, N, Z, seed=6, gen=2)
            Fd = torch.from_numpy(F).cuda()
            rank = torch.empty(20, 2 * N, dtype=torch.int32, device="cuda")
            sel = torch.empty(20, N, dtype=torch.int32, device="cuda")
            s = torch.cuda.current_stream().cuda_stream
            r.check(n.nsga3_set_counter(r.ctx, 2, s))
            torch.cuda.synchronize()
            for k in range(20):
                if k % 5 == 0:
                    _busy(torch, side, x)
                r.check(n.nsga3_select(r.ctx, Fd.data_ptr(), rank[k].data_ptr(), sel[k].data_ptr(), s))
            torch.cuda.synchronize()
            assert r.sync() == 0
            assert (rank.cpu().numpy() == ref["rank"]).all() and (sel.cpu().numpy() == ref["selected"]).all()


@pytest.mark.parametrize("m,d,N,p1", [(3, 400, 92, 12), (8, 27, 1000, 4)])
def test_generations_beside_other_work(torch, m, d, N, p1):
    from paper_2504_06067_gb300 import native as n
    x = torch.rand(1 << 24, device="cuda")
    side = torch.cuda.Stream()
    W = wl.objective_weights(m, 2)
    out = []
    for busy in (False, True):
        with Run(n, m, d, N, p1, seed=8, W=W) as r:
            r.check(n.nsga3_init(r.ctx, None))
            r.sync()
            for _ in range(5):
                if busy:
                    _busy(torch, side, x)
                r.check(n.nsga3_run(r.ctx, 4, None))
            assert r.sync() == 0
            out.append(r.population())
            torch.cuda.synchronize()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
