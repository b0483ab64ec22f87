"""Products on the tensor cores are as accurate row by row as the FP64 kernels': right-hand sides whose entries differ by
many orders of magnitude, unit vectors and columns of zeros."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


def _columns(x, seed):
    """Eight right-hand sides for the points x."""
    N = x.shape[0]
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((N, 8))
    X[:, 1] = 0
    X[N // 3, 1] = 1.0                                   # a unit vector: a column of the matrix
    X[:, 2] *= 10.0 ** rng.uniform(-20, 0, N)            # every size
    X[:, 3] *= np.where(x[:, 0] < 0.1, 1.0, 1e-15)       # large in one region, small in the others
    X[:, 4] = 0
    X[:, 5] *= 10.0 ** (-12 * x[:, -1])                  # falling along an axis
    X[:, 6] = np.abs(X[:, 6])
    X[:, 7] = np.where(np.arange(N) == N - 1, 1.0, 1e-18)
    return X


@pytest.mark.parametrize("N,d,ell", [
    (3000, 2, 0.1),     # ragged last row block
    (4096, 3, 0.2),
    (3073, 1, 0.02),    # entries down to exp(-50)
    (5000, 3, 0.05),
])
def test_kernel_product_row_by_row(T, N, d, ell):
    """The bound of the FP64 kernel: entries within 4 2^-52 (1 + z) of exp(-z) on either side, sums of N terms."""
    import torch
    ctx = T.Context(0)
    x = inputs.points(N, d, N)
    z = np.sqrt(((x[:, None, :] - x[None, :, :]) ** 2).sum(-1)) / ell
    A = np.exp(-z) + 1e-3 * np.eye(N)
    X = _columns(x, N)
    W = A * 2 * (N + 4 * (1 + z) + 4) * 2.0 ** -52
    for cols in ([0, 1, 2, 3, 4, 5, 6, 7], [1], [0, 2], [6, 3, 7]):
        g = ctx.kernel_matvec(x, ell, 1e-3, T.fortran(torch.tensor(X[:, cols], device="cuda:0"))).cpu().numpy()
        err, tol = np.abs(g - A @ X[:, cols]), W @ np.abs(X[:, cols])
        assert np.all(err <= tol), (cols, (err > tol).sum(0))
    ctx.close()



def _tiles(M, tri):
    """(i, j, factors) of M's tiles: (A, None) on the diagonal (tri: its lower triangle), (U, V) below; and D."""
    inf, rk = M.info(), M.ranks()
    b, nb = inf["b"], inf["nb"]
    d, out = np.ones(nb * b), []
    for i in range(nb):
        A, dv = M.tile(i, i)
        if dv is not None:
            A = np.tril(A, -1) + np.eye(b)
            d[i * b:(i + 1) * b] = dv
        out.append((i, i, np.tril(A) if tri else A, None))
        out += [(i, j, *M.tile(i, j)) for j in range(i) if rk[i, j]]
    return out, b, d


def _product(tiles, b, X, rows, columns):
    """The sum of the tiles' products with X (rows: as they lie; columns: transposed) and that of the absolute values."""
    Y, B, Xa = np.zeros_like(X), np.zeros_like(X), np.abs(X)
    for i, j, U, V in tiles:
        s, q = slice(i * b, (i + 1) * b), slice(j * b, (j + 1) * b)
        Ua = np.abs(U)
        if V is None:
            Y[s] += (U if rows else U.T) @ X[s]
            B[s] += (Ua if rows else Ua.T) @ Xa[s]
            continue
        Va = np.abs(V)
        if rows:
            Y[s] += U @ (V.T @ X[q])
            B[s] += Ua @ (Va.T @ Xa[q])
        if columns:
            Y[q] += V @ (U.T @ X[s])
            B[q] += Va @ (Ua.T @ Xa[s])
    return Y, B


@pytest.mark.parametrize("N,d,b,eps,ldl,all_tc", [
    (3000, 3, 250, 1e-6, True, False),     # tiles and segments that end inside a step of 16
    (4100, 2, 514, 1e-6, False, False),    # ragged last tile
    (12000, 3, 500, 1e-6, True, True),     # the factor's products on the tensor cores too
    (13000, 3, 512, 1e-6, False, True),
])
def test_products_row_by_row(T, N, d, b, eps, ldl, all_tc):
    """The bound of the FP64 kernels (test_gpu_apply.py): n u (|D| + |U| |V|^T) |X| on either side, with n the number of
    terms."""
    import torch
    ctx = T.Context(0)
    o = T.default_opts(bs=16, seed=N)
    x = inputs.points(N, d, N)
    A = ctx.compress(x, b, eps, 0.1, 1e-3, o)
    F = A.copy()
    (F.ldlt if ldl else F.potrf)(eps, o)
    ta, _, _ = _tiles(A, False)
    tl, _, dv = _tiles(F, True)
    perm = A.perm()
    X = _columns(x, N)
    X[:, 4] = np.arange(N) < N // 4
    X[perm, 4] *= 10.0 ** -(np.arange(N) % b / b * 18.0)  # falling along a tile
    npad = dv.size
    n = npad + int(max(A.ranks().sum(), F.ranks().sum()))
    u = 2.0 ** -53
    for cols in ([0, 1, 2, 3, 4, 5, 6, 7], [7, 6, 5, 4, 3, 2, 1], [0] * 8, [1] * 8):
        Xp = np.zeros((npad, len(cols)))
        Xp[:N] = X[perm][:, cols]
        Z, ZB = _product(tl, b, Xp, False, True)
        D = dv[:, None]
        want = {
            "A": (A, T.OP_A, *_product(ta, b, Xp, True, True), 1),
            "L": (F, T.OP_L, *_product(tl, b, Xp, True, False), 1),
            "Lt": (F, T.OP_LT, Z, ZB, 1),
            "LLt": (F, T.OP_LLT, _product(tl, b, D * Z, True, False)[0], _product(tl, b, np.abs(D) * ZB, True, False)[1], 2),
        }
        for name, (M, op, Y, B, times) in want.items():
            l0 = ctx.launches()
            g = M.matvec(T.fortran(torch.tensor(X[:, cols], device="cuda:0")), op).cpu().numpy()[perm]
            if all_tc:
                assert ctx.launches() - l0 >= 7  # three or five without the tensor cores
            err, tol = np.abs(g - Y[:N]), 2 * times * n * u * B[:N]
            assert np.all(err <= tol), (name, cols, (err > tol).sum(0))
    ctx.close()
