"""Two host threads with a context each, on one stream: their launches of a kernel may ask for different amounts of
shared memory."""
import threading

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


def _both(work):
    """Runs work(0) and work(1) in a thread each, again and again; the first error of either is raised."""
    errors = []

    def loop(i):
        try:
            for _ in range(200):
                if errors:
                    return
                work(i)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=loop, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def test_solves_of_different_sizes(T):
    import torch
    ctx, F, B, want = [], [], [], []
    for N, b in ((512, 64), (2600, 1300)):
        ctx.append(T.Context(0))
        F.append(ctx[-1].compress(inputs.points(N, 2, N), b, 1e-4, 0.1, 1e-2).potrf(1e-4))
        B.append(T.fortran(torch.tensor(inputs.rhs(N, 8, N), device="cuda:0")))
        want.append(F[-1].solve(B[-1].clone()).cpu().numpy())
    last = [None, None]

    def solve(i):
        last[i] = F[i].solve(B[i].clone())

    _both(solve)
    for i in range(2):
        assert np.array_equal(last[i].cpu().numpy(), want[i])
        ctx[i].close()


def test_trimming_of_different_ranks(T):
    import torch
    ctx, tiles, want = [], [], []
    for b, r in ((64, 10), (256, 140)):
        ctx.append(T.Context(0))
        Q, B, _ = inputs.lowrank_tiles(2, b, r, seed=r)
        tiles.append([torch.tensor(np.ascontiguousarray(np.transpose(x, (0, 2, 1))), device="cuda:0") for x in (Q, B)])
        want.append([x.cpu().numpy() if hasattr(x, "cpu") else x for x in ctx[-1].trim_tiles(*tiles[-1], 1e-20)])
    got = [None, None]

    def trim(i):
        got[i] = ctx[i].trim_tiles(*tiles[i], 1e-20)

    _both(trim)
    for i in range(2):
        for x, y in zip(got[i], want[i]):
            assert np.array_equal(x.cpu().numpy() if hasattr(x, "cpu") else x, y)
        ctx[i].close()
