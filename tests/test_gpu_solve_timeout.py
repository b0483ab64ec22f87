"""A solve whose bounded device wait runs out is reported by the call that it belongs to, not by a later one.

No device wait runs out here: the word that a solve sets in that case is set from the host, in the allocation that a
factor's first solve makes after it has looked at the word."""
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


class _Allocations:
    """The library's device allocations from arm() on; the word is set in the one after `after` says true."""

    def __init__(self, T, monkeypatch):
        import torch
        self.ctx = T.Context(0)
        f = T._load().tlr_solve_wait_word
        f.restype, f.argtypes = C.POINTER(C.c_int), [C.c_void_p]
        self.word = f(self.ctx.h)
        self.after = None
        self.seen = []
        alloc = torch.cuda.caching_allocator_alloc

        def patched(nbytes, *a, **k):
            if self.after and self.after(self.seen):
                self.word[0] = 1
                self.after = None
            self.seen.append(int(nbytes))
            return alloc(nbytes, *a, **k)

        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", patched)

    def arm(self, after):
        self.seen, self.after = [], after


def test_pcg_reports_its_last_solve(T, monkeypatch):
    import torch
    h = _Allocations(T, monkeypatch)
    N = 700
    x = inputs.points(N, 2, 3)
    A = h.ctx.compress(x, 128, 1e-6, 0.1, 1e-2)
    F = A.copy().potrf(1e-2)
    B = T.fortran(torch.tensor(inputs.rhs(N, 1, 3), device="cuda:0"))
    h.arm(lambda seen: len(seen) == 5)  # its five work arrays; then the solve's own
    with pytest.raises(T.TLRError) as e:
        A.pcg(F, B, tol=1e-10, maxit=1)
    assert e.value.status == T.ERR_TIMEOUT and h.after is None
    assert h.word[0] == 0
    X, _, res = A.pcg(F, B, tol=1e-10, maxit=50)
    assert bool(torch.isfinite(X).all())
    h.ctx.close()


def test_a_served_request_reports_its_own_solve(T, monkeypatch):
    h = _Allocations(T, monkeypatch)
    N, nrhs = 1000, 3
    x, rhs = inputs.points(N, 2, 4), inputs.rhs(N, nrhs, 4)

    def served(tickets):
        out = {}
        while len(out) < len(tickets):
            h.ctx.progress()
            for t in tickets:
                got = None if t in out else h.ctx.poll(t, N, nrhs)
                if got is not None:
                    out[t] = got[0]["status"]
        return [out[t] for t in tickets]

    t = h.ctx.submit(x, 128, 1e-4, 0.1, 1e-2, rhs)
    h.arm(lambda seen: seen[-1:] == [8 * N * nrhs])  # the device copy of the right-hand sides; then the solve's own
    assert served([t]) == [T.ERR_TIMEOUT] and h.after is None
    assert h.word[0] == 0
    assert served([h.ctx.submit(x, 128, 1e-4, 0.1, 1e-2, rhs)]) == [T.OK]
    h.ctx.close()
