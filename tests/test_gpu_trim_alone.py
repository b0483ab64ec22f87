"""A tile's trimming is a function of the tile: alone or among others, and scaled by a power of two."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


def _trim(T, ctx, Q, B, eps):
    import torch
    dev = lambda A: torch.tensor(np.ascontiguousarray(np.transpose(A, (0, 2, 1))), device="cuda:0")  # noqa: E731
    Qo, Bo, rk = ctx.trim_tiles(dev(Q), dev(B), eps)
    return [(Qo[t, :rk[t]].cpu().numpy(), Bo[t, :rk[t]].cpu().numpy()) for t in range(len(rk))]


@pytest.mark.parametrize("b,r,counts", [
    (128, 57, (1, 24, 160)),   # clusters of eight, of four, single CTAs
    (192, 140, (1, 30)),       # eight and four
    (96, 50, (3, 160)),        # an even number of columns, two or more pairs to a lane group
    (64, 33, (1, 5)),          # always one CTA
])
def test_a_tile_alone_and_among_others(T, b, r, counts):
    """Every sum of a tile runs in an order fixed by its rank: the same bits however many tiles the call has."""
    ctx = T.Context(0)
    Q, B, _ = inputs.lowrank_tiles(max(counts), b, r, seed=b + r)
    got = [_trim(T, ctx, Q[:n], B[:n], 1e-6) for n in counts]
    for g in got[1:]:
        for (q0, b0), (q1, b1) in zip(got[0], g):
            assert np.array_equal(q0, q1) and np.array_equal(b0, b1)
    ctx.close()


@pytest.mark.parametrize("nt,b,r", [(2, 96, 40), (1, 128, 75), (24, 128, 57)])
@pytest.mark.parametrize("k", [-290, 300])
def test_powers_of_two_scale_the_result(T, nt, b, r, k):
    """2^k B has the singular values and vectors of B, the former times 2^k: no square leaves the range of FP64 that a
    column's norm (and its square) stays in."""
    ctx = T.Context(0)
    Q, B, _ = inputs.lowrank_tiles(nt, b, r, seed=b + r, smin=1e-6)
    for (q0, b0), (q1, b1) in zip(_trim(T, ctx, Q, B, 1e-5), _trim(T, ctx, Q, np.ldexp(B, k), np.ldexp(1e-5, k))):
        assert np.array_equal(q0, q1) and np.array_equal(np.ldexp(b0, k), b1)
    ctx.close()
