"""Values that the solve's waits and reductions turn on: equal columns of a wide solve, and numbers that stand for
"not written yet" inside the kernel."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


def _factor(T, ctx, N, d, b, ldl=False):
    F = ctx.compress(inputs.points(N, d, N), b, 1e-4, 0.1, 1e-2, T.default_opts(bs=16, seed=N))
    return F.ldlt(1e-4) if ldl else F.potrf(1e-4)


@pytest.mark.parametrize("N,d,b,ldl,nrhs", [
    (2048, 3, 512, True, 32),    # four teams, units of 16 rows x 8 columns
    (1600, 2, 512, False, 24),   # three teams, ragged last tile
    (2600, 2, 2100, False, 6),   # one team, units of 16 rows x 6 columns
    (1000, 3, 64, True, 3),      # units smaller than a warp's share of the reduction
])
def test_equal_columns_get_equal_bits(T, N, d, b, ldl, nrhs):
    """Every column of a group is summed in the same order, so equal right-hand sides give equal bits."""
    import torch
    ctx = T.Context(0)
    F = _factor(T, ctx, N, d, b, ldl)
    y = np.random.default_rng(N).standard_normal((N, 1))
    first = None
    for _ in range(3):
        g = F.solve(T.fortran(torch.tensor(np.repeat(y, nrhs, axis=1), device="cuda:0"))).cpu().numpy()
        assert np.array_equal(g, np.repeat(g[:, :1], nrhs, axis=1))
        first = g if first is None else first
        assert np.array_equal(g, first)
    ctx.close()


@pytest.mark.parametrize("N,d,b,ldl", [(1000, 2, 128, False), (2048, 3, 512, True)])
def test_special_numbers_in_the_right_hand_side(T, N, d, b, ldl):
    """NaN, infinities and the very NaN that marks an entry as not yet written run through the solve like any other
    number: it ends, the affected columns hold no finite nonsense in the affected rows, the others keep their bits."""
    import torch
    ctx = T.Context(0)
    F = _factor(T, ctx, N, d, b, ldl)
    perm = F.perm()
    first, last = perm[0], perm[N - 1]  # of the elimination order
    marker = np.array([0x7ff85a3c96e10f2d], dtype=np.uint64).view(np.float64)[0]
    Y = np.random.default_rng(N).standard_normal((N, 8))
    clean = F.solve(T.fortran(torch.tensor(Y, device="cuda:0"))).cpu().numpy()
    B = Y.copy()
    B[first, 1], B[first, 2], B[last, 3], B[last, 4], B[first, 6] = marker, np.nan, marker, np.nan, np.inf
    B[:, 7] = marker
    g = F.solve(T.fortran(torch.tensor(B, device="cuda:0"))).cpu().numpy()
    for c in (0, 5):
        assert np.array_equal(g[:, c], clean[:, c])
    for c in (1, 3):  # the marker is a NaN like any other
        assert np.array_equal(np.isnan(g[:, c]), np.isnan(g[:, c + 1]))
        assert np.isnan(g[last, c]) and np.isnan(g[first, c])
    assert not np.isfinite(g[first, 6]) and np.isnan(g[:, 7]).all()
    assert np.array_equal(F.solve(T.fortran(torch.tensor(Y, device="cuda:0"))).cpu().numpy(), clean)
    ctx.close()
