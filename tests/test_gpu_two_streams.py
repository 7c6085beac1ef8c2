"""Calls that only read a context, made on two streams without order between
them, to destinations that rows are staged for (device addresses off 4 bytes):
each gets its own rows."""
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


@pytest.mark.parametrize("d,N", [(200, 60000), (33, 514)])
def test_population_and_children_on_two_streams(n, d, N):
    import torch
    m = 3
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with Run(n, m, d, N, 3, seed=5, W=wl.objective_weights(m, 1)) as r:
        r.check(n.nsga3_init(r.ctx, None))
        r.check(n.nsga3_step(r.ctx, None))
        X, Xc = r.population()[0], r.children()[0]
        px = torch.zeros(4 * N * d + 8, dtype=torch.uint8, device="cuda")
        pc = torch.zeros(4 * N * d + 8, dtype=torch.uint8, device="cuda")
        for off in (1, 2, 3):
            px.zero_(), pc.zero_()
            torch.cuda.synchronize()
            r.check(n.nsga3_get_population(r.ctx, px[off:].data_ptr(), None, None, a.cuda_stream))
            r.check(n.nsga3_get_children(r.ctx, pc[off:].data_ptr(), None, b.cuda_stream))
            torch.cuda.synchronize()
            for t, want in ((px, X), (pc, Xc)):
                got = t[off:off + 4 * N * d].cpu().numpy().view(np.float32).reshape(N, d)
                assert np.array_equal(got, want)
