"""The blocks of samples that a construction or factorization forms ahead of their rounds stay within eight rounds per
slot (the most an operand samples at once), and one more where a request finds none free."""
import ctypes as C

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


@pytest.mark.parametrize("N,d,b,eps,slots", [
    (4096, 3, 128, 1e-6, 0),    # ranks from a few to above 100: requests of every size
    (4096, 3, 128, 1e-6, 5),    # few slots, refilled again and again
    (2048, 2, 64, 1e-4, 0),
])
def test_blocks_of_samples_are_bounded(T, N, d, b, eps, slots):
    ctx = T.Context(0)
    f = T._load().tlr_sample_rounds_per_slot
    f.restype, f.argtypes = C.c_double, [C.c_void_p]
    o = T.default_opts(bs=16, seed=N, max_slots=slots)
    A = ctx.compress(inputs.points(N, d, N), b, eps, 0.2, 1e-2, o)
    assert 0 < f(ctx.h) <= 9
    F = A.copy().potrf(eps, o)
    assert f(ctx.h) <= 9
    if slots:  # the factor of any number of slots is the same
        o.max_slots = 0
        G = A.copy().potrf(eps, o)
        assert np.array_equal(F.ranks(), G.ranks())
        for i in range(1, A.info()["nb"], 5):
            for x, y in zip(F.tile(i, i - 1), G.tile(i, i - 1)):
                assert np.array_equal(x, y)
    ctx.close()
