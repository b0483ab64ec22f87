"""Products with a whole matrix or factor (tlr_matvec) against the dense matrix of its exported tiles.

Tolerance: every output is a sum of products in some order, so its error is at most n u (|D| + |U| |V|^T) |X|
with n the number of terms of the two contractions (Higham, Section 3.1); applied twice for L L^T.
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


def _dense(M, tri):
    """The matrix of M's tiles in KD order and the same of the absolute factors (tri: lower block triangle,
    of the diagonal tiles the lower triangle)."""
    inf, rk = M.info(), M.ranks()
    b, nb = inf["b"], inf["nb"]
    D, P = np.zeros((nb * b, nb * b)), np.zeros((nb * b, nb * b))
    d = np.ones(nb * b)
    for i in range(nb):
        s = slice(i * b, (i + 1) * b)
        A, dv = M.tile(i, i)
        if dv is not None:
            A = np.tril(A, -1) + np.eye(b)
            d[s] = dv
        D[s, s] = np.tril(A) if tri else A
        P[s, s] = np.abs(D[s, s])
        for j in range(i):
            if not rk[i, j]:
                continue
            q = slice(j * b, (j + 1) * b)
            U, V = M.tile(i, j)
            D[s, q], P[s, q] = U @ V.T, np.abs(U) @ np.abs(V).T
            if not tri:
                D[q, s], P[q, s] = D[s, q].T, P[s, q].T
    return D, P, d


@pytest.mark.parametrize("N,d,b,eps,ldl", [
    (100, 2, 128, 1e-6, False),    # one tile, ragged
    (1024, 2, 128, 1e-6, False),   # row blocks shared by clusters
    (1000, 3, 64, 1e-4, True),     # ragged last tile
    (700, 2, 75, 1e-6, False),     # odd tile size: 8-byte loads
    (600, 2, 50, 1e-3, True),      # row blocks of 64 cut short
    (1500, 1, 48, 1e-2, False),    # 1D: rank-1 and rank-0 tiles
])
def test_products_match_the_exported_tiles(T, N, d, b, eps, ldl):
    import torch
    ctx = T.Context(0)
    o = T.default_opts(bs=16, seed=N)
    A = ctx.compress(inputs.points(N, d, N), b, eps, 0.1, 1e-2 if eps > 1e-5 else 1e-4, o)
    F = A.copy()
    (F.ldlt if ldl else F.potrf)(eps, o)
    DA, PA, _ = _dense(A, False)
    L, PL, dv = _dense(F, True)
    npad = DA.shape[0]
    perm = A.perm()
    u = 2.0 ** -53
    rng = np.random.default_rng(N)
    for nrhs in (1, 2, 3, 5, 7, 8, 9, 17):
        X = rng.standard_normal((N, nrhs))
        Xp = np.zeros((npad, nrhs))
        Xp[:N] = X[perm]
        n = npad + int(max(A.ranks().sum(), F.ranks().sum()))
        want = {
            "A": (A, T.OP_A, DA @ Xp, PA @ np.abs(Xp), 1),
            "L": (F, T.OP_L, L @ Xp, PL @ np.abs(Xp), 1),
            "Lt": (F, T.OP_LT, L.T @ Xp, PL.T @ np.abs(Xp), 1),
            "LLt": (F, T.OP_LLT, L @ (dv[:, None] * (L.T @ Xp)),
                    PL @ (np.abs(dv)[:, None] * (PL.T @ np.abs(Xp))), 2),
        }
        for name, (M, op, Y, B, times) in want.items():
            g = M.matvec(T.fortran(torch.tensor(X, device="cuda:0")), op).cpu().numpy()[perm]
            assert np.all(np.abs(g - Y[:N]) <= 2 * times * n * u * B[:N]), (name, nrhs)
    ctx.close()


@pytest.mark.parametrize("N,d,b,eps,ldl", [
    (3000, 3, 250, 1e-6, True),     # tiles and segments that end inside a step of 16
    (4100, 2, 514, 1e-6, False),
])
def test_products_of_several_columns_on_the_tensor_cores(T, N, d, b, eps, ldl):
    """Entries and coefficients are rounded to 2^-58 of their columns' bounds (at most twice the largest), so a term's
    error is at most 2^-55.4 of the largest |a| |x| of its row block: n u max(|A| |X|) in all per contraction.
    Columns that the digits cannot hold go through the FP64 kernels: they match the columns one by one."""
    import torch
    ctx = T.Context(0)
    o = T.default_opts(bs=16, seed=N)
    A = ctx.compress(inputs.points(N, d, N), b, eps, 0.1, 1e-3, o)
    F = A.copy()
    (F.ldlt if ldl else F.potrf)(eps, o)
    DA, PA, _ = _dense(A, False)
    L, PL, dv = _dense(F, True)
    perm = A.perm()
    u = 2.0 ** -53
    rng = np.random.default_rng(N)
    for nrhs, scale in ((7, 1.0), (8, 1e-200), (16, 1e200)):
        X = rng.standard_normal((N, nrhs)) * scale * 10.0 ** rng.uniform(-3, 0, nrhs)
        Xp = np.zeros((DA.shape[0], nrhs))
        Xp[:N] = X[perm]
        n = DA.shape[0] + int(max(A.ranks().sum(), F.ranks().sum()))
        want = {
            "A": (A, T.OP_A, DA @ Xp, PA @ np.abs(Xp), 1),
            "L": (F, T.OP_L, L @ Xp, PL @ np.abs(Xp), 1),
            "Lt": (F, T.OP_LT, L.T @ Xp, PL.T @ np.abs(Xp), 1),
            "LLt": (F, T.OP_LLT, L @ (dv[:, None] * (L.T @ Xp)),
                    PL @ (np.abs(dv)[:, None] * (PL.T @ np.abs(Xp))), 2),
        }
        for name, (M, op, Y, B, times) in want.items():
            g = M.matvec(T.fortran(torch.tensor(X, device="cuda:0")), op).cpu().numpy()[perm]
            assert np.all(np.abs(g - Y[:N]) <= 2 * times * n * u * B.max(0)), (name, nrhs)
    X = rng.standard_normal((N, 8))
    X[7, 1], X[N // 2, 2], X[N - 1, 3] = np.nan, np.inf, -np.inf
    X[:, 4] *= 1e-300
    X[:, 5] = 0
    for M, op in ((A, T.OP_A), (F, T.OP_L), (F, T.OP_LT), (F, T.OP_LLT)):
        g = M.matvec(T.fortran(torch.tensor(X, device="cuda:0")), op).cpu().numpy()
        for c in range(8):
            w = M.matvec(T.fortran(torch.tensor(X[:, c:c + 1], device="cuda:0")), op).cpu().numpy()[:, 0]
            assert np.array_equal(np.isnan(g[:, c]), np.isnan(w)), (op, c)
            f = np.isfinite(w)
            assert np.array_equal(g[~f, c], w[~f], equal_nan=True), (op, c)
            if f.any():
                assert np.allclose(g[f, c], w[f], rtol=0, atol=1e-12 * np.abs(w[f]).max()), (op, c)
    ctx.close()


@pytest.mark.parametrize("N,d,b,eps,ldl", [
    (100, 2, 128, 1e-6, False),     # one tile, ragged
    (1000, 3, 64, 1e-4, True),      # L D L^T, ragged last tile
    (700, 2, 75, 1e-6, False),      # odd tile size: columns on 8-byte boundaries
    (600, 2, 50, 1e-3, True),
    (1500, 1, 48, 1e-2, False),     # rank-1 and rank-0 tiles
    (1500, 2, 1100, 1e-4, False),   # columns longer than a thread's loads in flight
    (2600, 2, 2100, 1e-4, True),    # with 8 columns: longer than the staged vector
])
def test_solves_match_the_exported_factor(T, N, d, b, eps, ldl):
    """The solve applies explicit inverses of the diagonal tiles and sums of n terms, so its forward error is
    within n u cond(L D L^T) (Higham, Sections 8.1, 14.2); every column of every width on its own."""
    import torch
    ctx = T.Context(0)
    o = T.default_opts(bs=16, seed=N)
    F = ctx.compress(inputs.points(N, d, N), b, eps, 0.1, 1e-2 if eps > 1e-5 else 1e-4, o)
    (F.ldlt if ldl else F.potrf)(eps, o)
    L, _, dv = _dense(F, True)
    A = L @ (dv[:, None] * L.T)
    perm = F.perm()
    tol = A.shape[0] * 2.0 ** -52 * np.linalg.cond(A)
    rng = np.random.default_rng(N)
    Y = rng.standard_normal((N, 33))
    Yp = np.zeros((A.shape[0], 33))
    Yp[:N] = Y[perm]
    X = np.linalg.solve(A, Yp)[:N]
    for nrhs in (1, 2, 3, 5, 7, 8, 9, 33):
        B = T.fortran(torch.tensor(Y[:, :nrhs], device="cuda:0"))
        g = F.solve(B).cpu().numpy()[perm]
        err = np.linalg.norm(g - X[:, :nrhs], axis=0) / np.linalg.norm(X[:, :nrhs], axis=0)
        assert np.all(err <= tol), (nrhs, err.max(), tol)
    ctx.close()


@pytest.mark.parametrize("N,d,ell,scale,nrhs", [
    (1, 2, 0.1, 1.0, 1),
    (31, 1, 0.1, 1.0, 2),         # less than a warp's columns
    (33, 3, 0.2, 1.0, 3),
    (513, 2, 0.1, 1.0, 9),        # two groups of right-hand sides, a cluster of two
    (5000, 3, 0.2, 1.0, 8),       # a full cluster
    (700, 2, 0.01, 1.0, 5),       # extent above 64 ell: FP64 entries
    (700, 3, 30.0, 250.0, 4),     # off the unit box, on the grid
])
def test_kernel_product_matches_dense(T, N, d, ell, scale, nrhs):
    """Entries within 4 2^-52 (1 + z) of exp(-z) on either side, sums of N terms: the two sides differ by at most
    2 (N + 4 (1 + z) + 4) 2^-52 of the sum of |a_ij x_j|."""
    import torch
    ctx = T.Context(0)
    x = inputs.points(N, d, N) * scale - 0.3 * scale
    if N > 100:
        x[7] = x[60]  # coincident points
    X = np.random.default_rng(N).standard_normal((N, nrhs))
    g = ctx.kernel_matvec(x, ell, 1e-3, T.fortran(torch.tensor(X, device="cuda:0"))).cpu().numpy()
    z = np.sqrt(((x[:, None, :] - x[None, :, :]) ** 2).sum(-1)) / ell
    A = np.exp(-z) + 1e-3 * np.eye(N)
    B = (A * 2 * (N + 4 * (1 + z) + 4) * 2.0 ** -52) @ np.abs(X)
    assert np.all(np.abs(g - A @ X) <= B)
    ctx.close()


@pytest.mark.parametrize("N,d,ell,nrhs", [
    (3000, 2, 0.1, 1),            # ragged last row block
    (3073, 1, 0.02, 9),           # one row in the last block; two groups
    (4096, 3, 0.2, 8),
    (3300, 3, 0.01, 3),           # extent above 64 ell: FP64 entries
])
def test_large_kernel_products_match_dense(T, N, d, ell, nrhs):
    """As above, plus the fixed-point rounding of entries (2^-57) and right-hand sides (2^-58 of a bound of at most twice
    the largest): N 2^-55 of the largest."""
    import torch
    ctx = T.Context(0)
    x = inputs.points(N, d, N)
    x[7] = x[60]  # coincident points
    z = np.sqrt(((x[:, None, :] - x[None, :, :]) ** 2).sum(-1)) / ell
    A = np.exp(-z) + 1e-3 * np.eye(N)
    rng = np.random.default_rng(N)
    for scale in (1.0, 1e-150, 1e200, 1e-305):
        X = rng.standard_normal((N, nrhs)) * scale * 10.0 ** rng.uniform(-2, 0, nrhs)
        g = ctx.kernel_matvec(x, ell, 1e-3, T.fortran(torch.tensor(X, device="cuda:0"))).cpu().numpy()
        B = (A * 2 * (N + 4 * (1 + z) + 4) * 2.0 ** -52) @ np.abs(X) + N * 2.0 ** -55 * np.abs(X).max(0)
        assert np.all(np.abs(g - A @ X) <= B), scale
    X = np.abs(rng.standard_normal((N, nrhs)))
    X[N // 2, 0] = np.inf
    if nrhs > 1:
        X[N - 1, 1] = np.nan
    g = ctx.kernel_matvec(x, ell, 1e-3, T.fortran(torch.tensor(X, device="cuda:0"))).cpu().numpy()
    want = A @ X
    assert np.array_equal(np.isnan(g[:, 1:]), np.isnan(want[:, 1:]))
    assert np.isinf(g[:, 0]).all() and np.all(g[:, 0] > 0)
    f = np.isfinite(want)
    assert np.allclose(g[f], want[f], rtol=1e-10, atol=0)
    ctx.close()


def test_kernel_product_of_non_finite_points_is_nan(T):
    import torch
    ctx = T.Context(0)
    x = inputs.points(100, 2, 3)
    x[41, 1] = np.nan
    g = ctx.kernel_matvec(x, 0.1, 1e-3, T.fortran(torch.ones((100, 2), dtype=torch.float64, device="cuda:0")))
    assert bool(torch.isnan(g).all())  # every row sums the entry with point 41
    ctx.close()
