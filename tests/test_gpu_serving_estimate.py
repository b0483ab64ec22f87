"""The serving queue's estimate of a request's device bytes counts the work vectors of its solve."""
import ctypes as C

import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


@pytest.mark.parametrize("N,d,b,eps,ldl,nrhs", [
    (4096, 2, 128, 1e-6, False, 32),
    (4000, 2, 64, 1e-6, True, 17),
    (4096, 2, 128, 1e-6, False, 40),
    (4096, 2, 128, 1e-6, False, 1),
])
def test_estimate_counts_the_solve(T, N, d, b, eps, ldl, nrhs, monkeypatch):
    """Right-hand sides add at least their copy and what a solve of them allocates (2D ranks at 1e-6 stay below the
    estimate's mean rank of 18 for these tiles)."""
    import torch
    f = T._load().tlr_request_footprint
    f.restype, f.argtypes = C.c_size_t, [C.POINTER(T.Request)]

    def estimate(n):
        return f(C.byref(T.Request(None, N, d, T.Kernel(0, 0.1, 1e-2), b, eps, int(ldl), n, None, T.default_opts())))

    ctx = T.Context(0)
    F = ctx.compress(inputs.points(N, d, N), b, eps, 0.1, 1e-2)
    (F.ldlt if ldl else F.potrf)(eps)
    assert F.info()["mean_rank"] <= 18
    sizes = []
    alloc = torch.cuda.caching_allocator_alloc
    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", lambda n, *a, **k: (sizes.append(int(n)), alloc(n, *a, **k))[1])
    F.solve(T.fortran(torch.tensor(inputs.rhs(N, nrhs, 1), device="cuda:0")))
    monkeypatch.undo()
    assert len(sizes) == 2  # the step list (kept small) and the vectors
    assert estimate(nrhs) - estimate(0) >= max(sizes) + 8 * N * nrhs
    ctx.close()
