"""Rows of the decision vectors stay where they were written (index lists say
which row holds which individual): every call that reads or replaces the
population sees the same individuals whatever the order of the calls, for
widths with and without 16-byte rows and for host and device destinations."""
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


# (m, d, N): ragged and 16-byte row widths, one merged block and several, m > 10
SHAPES = [(3, 12, 92), (3, 7, 2), (5, 33, 130), (2, 1, 514), (10, 40, 600), (16, 21, 140)]


@pytest.mark.parametrize("m,d,N", SHAPES)
def test_population_calls_in_any_order(n, m, d, N):
    import torch
    W = wl.objective_weights(m, 1)
    with Run(n, m, d, N, 3 if m <= 10 else 1, seed=5, W=W) as r:
        r.check(n.nsga3_init(r.ctx, None))
        for g in range(3):
            X, F, rank = r.population()
            r.check(n.nsga3_step(r.ctx, None))
            Xc, Fc = r.children()
            Xn, Fn, rn = r.population()
            # the next parents are merged individuals, in merged order
            RX, RF = np.vstack([X, Xc]), np.vstack([F, Fc])
            at = -1
            for p in range(N):
                at = next(i for i in range(at + 1, 2 * N)
                          if np.array_equal(RX[i], Xn[p]) and np.array_equal(RF[i], Fn[p]))
            # a device destination (offset by one float: rows off 16 bytes) and a pinned one
            dev = torch.empty(N * d + 1, device="cuda")[1:]
            r.check(n.nsga3_get_population(r.ctx, dev.data_ptr(), None, None, None))
            pin = torch.empty(N, d, pin_memory=True)
            r.check(n.nsga3_get_children(r.ctx, pin.data_ptr(), None, None))
            assert r.sync() == 0
            assert np.array_equal(dev.cpu().numpy().reshape(N, d), Xn)
            assert np.array_equal(pin.numpy(), Xc)
        # replacing the parents keeps the last children
        Xs = wl.population(N, d, seed=3)
        src = torch.from_numpy(Xs).cuda()
        for ptr in (Xs.ctypes.data, src.data_ptr()):
            r.check(n.nsga3_set_population(r.ctx, ptr, Fn.ctypes.data, rn.ctypes.data, None))
            assert np.array_equal(r.children()[0], Xc) and np.array_equal(r.children()[1], Fc)
            X2, F2, r2 = r.population()
            assert np.array_equal(X2, Xs) and np.array_equal(F2, Fn) and np.array_equal(r2, rn)
            # new children leave the parents, also twice in a row
            r.check(n.nsga3_vary(r.ctx, None))
            r.check(n.nsga3_vary(r.ctx, None))
            Xc, Fc = r.children()
            assert np.array_equal(r.population()[0], Xs)


@pytest.mark.parametrize("shape", [(3, 2, 3), (3, 130, 7), (5, 1100, 8), (4, 514, 33), (12, 90, 13)])
def test_outputs_beside_the_rows(n, shape):
    """Rows, objectives and ranks written by one launch: device buffers, device
    buffers of odd addresses, host buffers and each of them left out give the
    same values, and nothing past their ends."""
    import torch
    m, N, d = shape
    W = wl.objective_weights(m, 3)
    with Run(n, m, d, N, 1, seed=4, W=W) as r:
        r.check(n.nsga3_init(r.ctx, None))
        r.check(n.nsga3_run(r.ctx, 3, None))
        X, F, rank = r.population()
        Xc, Fc = r.children()
        for off in (0, 1, 3):
            bx = torch.full((N * d + 8,), -7.0, device="cuda")
            bf = torch.full((N * m + 8,), -7.0, device="cuda")
            br = torch.full((N + 8,), -7, device="cuda", dtype=torch.int32)
            torch.cuda.synchronize()
            for what in (7, 1, 2, 4, 6):
                p = [t[off:].data_ptr() if what >> k & 1 else None for k, t in enumerate((bx, bf, br))]
                r.check(n.nsga3_get_population(r.ctx, p[0], p[1], p[2], None))
                r.check(r.sync())
            for t, a in ((bx, X), (bf, F), (br, rank)):
                h = t.cpu().numpy()
                assert np.array_equal(h[off:off + a.size], a.ravel())
                assert (h[:off] == -7).all() and (h[off + a.size:] == -7).all()
            r.check(n.nsga3_get_children(r.ctx, bx[off:].data_ptr(), bf[off:].data_ptr(), None))
            r.check(r.sync())
            assert np.array_equal(bx[off:off + N * d].cpu().numpy(), Xc.ravel())
            assert np.array_equal(bf[off:off + N * m].cpu().numpy(), Fc.ravel())
