"""The work that users of this framework have it do, as cases to be measured.

A user holds points of a spatial-statistics problem (uniform in the unit square or cube, exponential
covariance kernel with a small nugget), builds the tile-low-rank covariance matrix, and then applies it,
factors it, solves with the factor, takes its log-determinant, trims its ranks or uses a cheap factor as
a preconditioner.  Sizes, tolerances and options are those of the framework's own workloads: 2D
N = 4096 (b = 256) to N = 131072 (b = 1024), correlation length 0.1; 3D N = 32768 (b = 512, ARA blocks of
32), correlation length 0.2; batches of matrices of 2048 to 16384 points; eps from 1e-2 to 1e-8.

Each case is a dict of plain values; "kind" says which calls a pass makes:

  apply      Y = A X with the compressed matrix (the operator product of iterative methods)
  apply_llt  Y = L (D) L^T X with the factor (the product of the backward-error check)
  solve      X = F^{-1} B with a resident factor (the follow-up solves of a service)
  kernel     Y = K X with the exact kernel matrix, formed on the fly (residuals, error checks)
  construct  compression of the kernel matrix from host points, then one product with it
  likelihood the whole evaluation: construction, factorization, solve, log-determinant
  batch      factorization of several matrices together, then a solve with each
  trim       ARA -> SVD rank trimming of a compressed matrix, then one product with it
  pcg        conjugate gradients on an accurate matrix, preconditioned by a low-accuracy factor
"""
import functools
import math

import numpy as np
import torch

import paper_2108_11932_gb300 as tlr

NUGGET = 1e-4


@functools.lru_cache(maxsize=1)
def _context():
    """The library context of the process: a program makes one and keeps it."""
    return tlr.Context(0)


def _case(kind, N, d, b, eps, nrhs, bs=16, ldl=False, mixed=False, count=1, **more):
    return {"kind": kind, "N": N, "d": d, "b": b, "bs": bs, "eps": eps, "ell": 0.1 if d == 2 else 0.2, "nrhs": nrhs,
            "ldl": ldl, "mixed": mixed, "count": count, **more}


def listed():
    return [
        # one product with a small compressed matrix: an iteration of a Krylov method on a small field
        dict(_case("apply", 4096, 2, 256, 1e-6, 1), name="apply_2d_4k"),
        # a block of probe vectors through the largest matrix (stochastic trace estimates, samples)
        dict(_case("apply", 131072, 2, 1024, 1e-6, 8), name="apply_2d_131k_8"),
        # the factor's own product in 3D, ragged last tile: the power iteration of the error check
        dict(_case("apply_llt", 20011, 3, 512, 1e-4, 1, bs=32), name="apply_llt_3d_20k"),
        # a prediction from a small resident factor
        dict(_case("solve", 4096, 2, 256, 1e-6, 1), name="solve_2d_4k"),
        # a prediction from the largest resident factor
        dict(_case("solve", 131072, 2, 1024, 1e-6, 1), name="solve_2d_131k"),
        # many right-hand sides at once through a 3D L D L^T factor with a ragged last tile
        dict(_case("solve", 20011, 3, 512, 1e-4, 32, bs=32, ldl=True), name="solve_ldl_3d_20k_32"),
        # the exact product behind residuals and error estimates
        dict(_case("kernel", 32768, 3, 512, 1e-4, 4), name="kernel_3d_33k_4"),
        # building a 3D matrix from host points in mixed precision, ragged
        dict(_case("construct", 30011, 3, 512, 1e-4, 1, bs=32, mixed=True), name="construct_3d_30k"),
        # the headline evaluation
        dict(_case("likelihood", 131072, 2, 1024, 1e-6, 1), name="likelihood_2d_131k"),
        # a sweep over hyper-parameters: small matrices of mixed sizes factored together
        dict(_case("batch", 8192, 2, 256, 1e-6, 1, count=8), name="batch_2d_8k_x8"),
        # rank trimming of a compressed matrix before it is stored
        dict(_case("trim", 16384, 2, 512, 1e-6, 1), name="trim_2d_16k"),
        # an accurate solve through a cheap preconditioner
        dict(_case("pcg", 32768, 2, 512, 1e-8, 1, peps=1e-4), name="pcg_2d_33k"),
    ]


def _size(rng, lo, hi):
    """A size of the range, log-uniform; one in two is odd."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n | 1 if rng.random() < 0.5 else (n + 255) // 256 * 256


def draw(rng):
    kind = rng.choice(["apply", "apply_llt", "solve", "solve", "kernel", "construct", "likelihood", "batch", "trim", "pcg"])
    d = rng.choice([2, 3])
    top = {"apply": 100000, "apply_llt": 65536, "solve": 65536, "kernel": 40000, "construct": 65536, "likelihood": 65536,
           "batch": 8192, "trim": 16384, "pcg": 32768}[kind]
    if d == 3:  # ranks, and with them the work per point, are several times those of 2D
        top = min(top, 4096 if kind == "trim" else 32768)
    N = _size(rng, 2048, top)
    b = 1024 if N >= 60000 else 512 if N >= 16384 else 256
    eps = rng.choice([1e-2, 1e-4, 1e-6])
    if d == 3 and N > 16384:
        eps = max(eps, 1e-4)
    if d == 3 and kind in ("apply_llt", "solve", "likelihood", "batch"):
        eps = min(eps, 1e-4)
    nrhs = {"apply": rng.randint(1, 16), "apply_llt": rng.randint(1, 8), "solve": rng.randint(1, 32),
            "kernel": rng.randint(1, 8), "likelihood": rng.randint(1, 32), "pcg": rng.randint(1, 4)}.get(kind, 1)
    c = _case(kind, N, d, b, eps, nrhs, bs=rng.choice([16, 32]) if d == 3 else 16,
              ldl=kind in ("apply_llt", "solve", "likelihood", "batch") and rng.random() < 0.4,
              mixed=kind in ("construct", "likelihood") and eps >= 1e-4 and rng.random() < 0.4,
              count=rng.randint(2, 12) if kind == "batch" else 1)
    if kind == "pcg":
        c["eps"], c["peps"] = 1e-8 if d == 2 else 1e-6, 1e-4
    return c


# ------------------------------------------------------------------ inputs
def _sizes(case):
    """Points of each matrix: a batch spreads them over N/4 .. N in whole tiles."""
    n = case["count"]
    if case["kind"] != "batch":
        return [case["N"]]
    b = case["b"]
    return [max(b, int(case["N"] * (0.25 + 0.75 * (m + 1) / n)) // b * b) for m in range(n)]


def _points(case, seed):
    rng = np.random.default_rng(seed)
    return [rng.random((n, case["d"])) for n in _sizes(case)]


def _rhs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    return [tlr.fortran(torch.randn((n, case["nrhs"]), dtype=torch.float64, device="cuda", generator=g))
            for n in _sizes(case)]


def _opts(case, seed, **more):
    return tlr.default_opts(bs=case["bs"], seed=seed, precision=tlr.PREC_MIXED if case["mixed"] else tlr.PREC_FP64, **more)


def _factor(A, case, seed):
    o = _opts(case, seed)
    return A.ldlt(case["eps"], o) if case["ldl"] else A.potrf(case["eps"], o)


def prepare(case, seed):
    ctx = _context()
    s = {"case": case, "seed": seed, "pts": _points(case, seed), "rhs": _rhs(case, seed)}
    kind = case["kind"]
    if kind in ("kernel", "construct", "likelihood"):
        return s
    s["A"] = [ctx.compress(x, case["b"], case["eps"], case["ell"], NUGGET, _opts(case, seed)) for x in s["pts"]]
    if kind in ("apply_llt", "solve"):
        s["F"] = _factor(s.pop("A")[0], case, seed)
    elif kind == "pcg":
        e = case["peps"]
        M = ctx.compress(s["pts"][0], case["b"], e, case["ell"], NUGGET, _opts(case, seed))
        s["F"] = M.potrf(e, _opts(case, seed, compensation=tlr.COMP_SHIFT, shift=e))
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    case, seed, ctx = state["case"], state["seed"], _context()
    kind, X = case["kind"], state["rhs"][0]
    if kind == "apply":
        return state["A"][0].matvec(X, tlr.OP_A)
    if kind == "apply_llt":
        return state["F"].matvec(X, tlr.OP_LLT)
    if kind == "solve":
        return state["F"].solve(X.clone())  # solved in place: the right-hand sides stay for the next pass
    if kind == "kernel":
        return ctx.kernel_matvec(state["pts"][0], case["ell"], NUGGET, X)
    if kind == "construct":
        A = ctx.compress(state["pts"][0], case["b"], case["eps"], case["ell"], NUGGET, _opts(case, seed))
        return A.matvec(X, tlr.OP_A)
    if kind == "likelihood":
        A = ctx.compress(state["pts"][0], case["b"], case["eps"], case["ell"], NUGGET, _opts(case, seed))
        F = _factor(A, case, seed)
        Y = F.solve(X.clone())
        logdet, sign = F.logdet()
        return Y, np.float64(logdet), sign
    if kind == "batch":
        F = [A.copy() for A in state["A"]]
        status = ctx.factor_batch(F, case["eps"], _opts(case, seed), ldl=case["ldl"])
        return [f.solve(B.clone()) for f, B in zip(F, state["rhs"])], status
    if kind == "trim":
        return state["A"][0].copy().trim(case["eps"]).matvec(X, tlr.OP_A)
    X, iterations, _ = state["A"][0].pcg(state["F"], X, tol=1e-6, maxit=300)
    return X, iterations


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    nrhs, b, d = case["nrhs"], case["b"], case["d"]
    r = max(1.0, (2.7 if d == 2 else 12.5) * -math.log10(case["eps"]))  # mean rank of the off-diagonal tiles
    by = fl = 0.0
    for n in _sizes(case):
        nb = -(-n // b)
        pairs = nb * (nb - 1) / 2
        vec = 16.0 * n * nrhs
        low = 2 * pairs * b * r                                          # entries of the U and V factors
        tri = nb * b * (b + 1) / 2                                       # entries of the (symmetric) diagonal tiles
        use = (8 * (low + tri) + vec, 2 * nrhs * (2 * low + nb * b * b))   # one product or one solve
        make = (8 * (n * d + low + tri), pairs * b * b * (30.0 + 4 * r + 2 * case["bs"]) + nb * b * b * 30.0)
        fact = (16 * (low + tri), pairs * (nb / 3) * 12.0 * b * r * r + nb * b ** 3 / 3)
        kind = case["kind"]
        for w, times in ((use, 1 if kind not in ("kernel", "pcg") else 0), (make, kind in ("construct", "likelihood")),
                         (fact, kind in ("likelihood", "batch")), (use, 12 * (kind == "pcg"))):
            by += w[0] * times
            fl += w[1] * times
        if kind == "kernel":
            by += 8 * n * d + vec
            fl += n * n * (3.0 * d + 25 + 2 * nrhs)
        if kind == "trim":
            by += 16 * low
            fl += pairs * (8 * b * r * r + 30 * r ** 3)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ the same in plain 64-bit torch
def _kernel_rows(x, lo, hi, ell):
    K = torch.exp(torch.cdist(x[lo:hi], x, compute_mode="donot_use_mm_for_euclid_dist") * (-1.0 / ell))
    i = torch.arange(lo, hi, device=x.device)
    K[i - lo, i] = 1.0 + NUGGET
    return K


def _kernel_product(x, X, ell):
    step = max(1, (1 << 27) // x.shape[0])
    return torch.cat([_kernel_rows(x, lo, min(lo + step, x.shape[0]), ell) @ X for lo in range(0, x.shape[0], step)])


def _kernel_solve(x, B, ell, logdet=False):
    L = torch.linalg.cholesky(_kernel_rows(x, 0, x.shape[0], ell))
    Y = torch.cholesky_solve(B, L)
    return (Y, 2 * L.diagonal().log().sum()) if logdet else Y


def exact(case, seed):
    kind, ell = case["kind"], case["ell"]
    pts = [torch.tensor(x, device="cuda") for x in _points(case, seed)]
    rhs = _rhs(case, seed)
    if kind in ("apply", "apply_llt", "kernel", "construct", "trim"):
        return _kernel_product(pts[0], rhs[0], ell)
    # solves: the dense factorization fits the time up to about 33,000 points; at eps = 1e-2 the
    # method's own truncation is as large as the solution's digits
    if case["eps"] > 1e-3 or case["N"] > 33000:
        return None
    if kind == "solve":
        return _kernel_solve(pts[0], rhs[0], ell)
    if kind == "likelihood":
        Y, logdet = _kernel_solve(pts[0], rhs[0], ell, logdet=True)
        return Y, np.float64(logdet.item()), None
    if kind == "batch":
        return [_kernel_solve(x, B, ell) for x, B in zip(pts, rhs)], None
    return _kernel_solve(pts[0], rhs[0], ell), None
