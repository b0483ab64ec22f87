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
