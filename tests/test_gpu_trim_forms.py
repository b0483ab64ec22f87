"""The launch forms of the rank trimming (one CTA, clusters of four and eight, R^T in global memory, single-CTA
tiles beside the clusters) against numpy's singular values."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


@pytest.mark.parametrize("nt,b,r", [
    (3, 96, 48),     # the highest rank of a single CTA
    (2, 96, 49),     # the lowest of a cluster (of eight: few tiles), an odd number of columns
    (24, 128, 57),   # enough tiles for clusters of four
    (160, 96, 50),   # more tiles of one rank than clusters fill the GPU with: one CTA each
    (1, 512, 480),   # R^T larger than eight CTAs' shared memory
])
def test_singular_values_and_products(T, nt, b, r):
    """One-sided Jacobi and Householder QR are backward stable: singular values within a modest multiple of
    b u smax (here 64) and the untrimmed product to the same."""
    import torch
    ctx = T.Context(0)
    Q, B, s = inputs.lowrank_tiles(nt, b, r, seed=b + r)
    dev = lambda A: torch.tensor(np.ascontiguousarray(np.transpose(A, (0, 2, 1))), device="cuda:0")  # noqa: E731
    eps = 3e-5
    Qo, Bo, rk = ctx.trim_tiles(dev(Q), dev(B), eps)
    Qo, Bo = (np.transpose(x.cpu().numpy(), (0, 2, 1)) for x in (Qo, Bo))
    tol = 64 * b * 2.0 ** -53 * s.max()
    for t in range(nt):
        sv = np.linalg.svd(B[t], compute_uv=False)
        q = int(rk[t])
        assert sv[q - 1] > eps - tol and (q == r or sv[q] <= eps + tol), t
        assert np.abs(np.linalg.norm(Bo[t][:, :q], axis=0) - sv[:q]).max() <= tol
        assert np.linalg.norm(Q[t] @ B[t].T - Qo[t][:, :q] @ Bo[t][:, :q].T, 2) <= (sv[q] if q < r else 0) + tol
    ctx.close()


def test_a_matrix_with_low_and_high_ranks(T):
    """Both streams: every tile of the trimmed matrix within eps of the untrimmed one, none of higher rank."""
    ctx = T.Context(0)
    eps = 1e-6
    A = ctx.compress(inputs.points(2048, 2, 5), 256, eps, 0.1, 1e-4, T.default_opts(seed=5))
    R = A.ranks()
    assert R[R > 0].min() <= 48 < R.max()
    M = A.copy().trim(eps)
    S = M.ranks()
    for i in range(A.info()["nb"]):
        for j in range(i):
            U, V = A.tile(i, j)
            Ut, Vt = M.tile(i, j)
            assert S[i, j] <= R[i, j]
            assert np.linalg.norm(U @ V.T - Ut @ Vt.T, 2) <= eps * (1 + 1e-6), (i, j)
    ctx.close()
