"""The calls that a user of this library makes, as timed cases.

Two kinds of work are measured, both through the public Python front end:
one application of the preconditioner M^{-1} (``Gemslr.apply``,
``GemslrBatch.apply``: what a caller with a Krylov method of their own uses)
and whole FGMRES solves (``Gemslr.solve``, ``GemslrBatch.solve``).  Operators
are finite-difference stencils on 2-D and 3-D grids, right-hand sides uniform
in [-1, 1).  A state holds the set-up handle and the right-hand sides on the
GPU; every pass applies or solves once.

A case is a dict of plain values:
  kind       "apply", "solve", "batch_apply" or "batch_solve"
  dims       grid, "nx x ny (x nz)" (single systems)
  beta       convection; sigma: diagonal shift -sigma h^-2
  nlev, p    levels and subdomains per level; local_from: first level whose
             blocks take the local multicolour order (-1: none)
  ilu, tau, lfil, rank, precision, shift: set-up options
  nrhs       right-hand sides (of every system in a batch)
  restart    FGMRES cycle length (solves run to a relative residual of 1e-8)
  count, lo, hi, sysseed: batches of `count` systems with sides in [lo, hi]
"""
import functools
import math

import numpy as np
import torch

import gemslr_inputs as gi
from paper_2205_03224_gb300 import Gemslr, GemslrBatch, partition_geometric

RTOL = 1e-8


def _single(name, kind, dims, nlev, p, ilu, tau, lfil, rank, precision, beta=0.0, sigma=0.0, local_from=-1,
            shift=0.0, nrhs=1, restart=50):
    c = dict(name=name, kind=kind, dims=dims, beta=beta, sigma=sigma, nlev=nlev, p=p, local_from=local_from, ilu=ilu,
             tau=tau, lfil=lfil, rank=rank, precision=precision, shift=shift, nrhs=nrhs, restart=restart)
    if name is None:
        del c["name"]
    return c


def _batch(name, kind, count, lo, hi, nlev, p, tau, lfil, rank, nrhs, sysseed, restart=50):
    c = dict(name=name, kind=kind, count=count, lo=lo, hi=hi, sysseed=sysseed, nlev=nlev, p=p, ilu="ilut", tau=tau,
             lfil=lfil, rank=rank, nrhs=nrhs, restart=restart)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the smallest call: one application on a 2-D model problem of 1,024
        # unknowns, where launches and latency are everything
        _single("apply_fp64_32sq", "apply", "32x32", 2, 4, "ilu0", 0.0, 0, 8, "fp64"),
        # the same problem solved: the smallest whole solve
        _single("solve_fp64_32sq", "solve", "32x32", 2, 4, "ilu0", 0.0, 0, 8, "fp64", restart=30),
        # the 3-D model problem of the benchmark, applied in the plain FP64
        # path (the parity reference) and in mixed precision (the default for speed)
        _single("apply_fp64_64cubed", "apply", "64x64x64", 4, 64, "ilut", 1e-3, 10, 32, "fp64", beta=0.1,
                local_from=1),
        _single("apply_mixed_64cubed", "apply", "64x64x64", 4, 64, "ilut", 1e-3, 10, 32, "mixed", beta=0.1,
                local_from=1),
        # the benchmark's solve: time to 1e-8 in mixed precision
        _single("solve_mixed_64cubed", "solve", "64x64x64", 4, 64, "ilut", 1e-3, 10, 32, "mixed", beta=0.1,
                local_from=1),
        # an FP64 solve of an odd box with several right-hand sides, a loose
        # factorisation and a small correction, blocks in ascending order
        _single("solve_fp64_odd_3rhs", "solve", "45x38x29", 3, 16, "ilut", 1e-2, 5, 5, "fp64", beta=0.4, nrhs=3),
        # the largest single system: the 128^3 shifted operator, rank 64
        _single("apply_mixed_128cubed", "apply", "128x128x128", 4, 64, "ilut", 1e-3, 10, 64, "mixed", sigma=0.05,
                local_from=1),
        # few large subdomains: block vectors that do not fit in shared memory
        _single("apply_fp64_240sq", "apply", "240x240", 2, 2, "ilu0", 0.0, 0, 4, "fp64", beta=0.5),
        # the complex diagonal shift for an indefinite operator: application and solve
        _single("apply_complex_48cubed", "apply", "48x48x48", 4, 64, "ilut", 1e-3, 10, 32, "fp64", sigma=0.05,
                local_from=1, shift=0.05),
        _single("solve_complex_32cubed", "solve", "32x32x32", 4, 8, "ilut", 1e-3, 10, 32, "fp64", sigma=0.05,
                shift=0.05, restart=60),
        # the batched benchmark: 96 uneven systems with 8 right-hand sides each
        _batch("batch_solve_96x8", "batch_solve", 96, 16, 48, 3, 8, 1e-3, 10, 16, 8, 3),
        # a small batch of small systems with an odd number of right-hand sides
        _batch("batch_apply_24x3", "batch_apply", 24, 6, 16, 3, 4, 1e-3, 10, 6, 3, 7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds: sizes spread over their logarithm, odd boxes, every option in use."""
    kind = rng.choice(["apply", "apply", "apply", "solve", "solve", "batch_apply", "batch_solve"])
    if kind.startswith("batch"):
        hi = rng.randint(12, 40)
        return _batch(None, kind, _log_int(rng, 3, 48), rng.randint(6, max(7, hi // 2)), hi, rng.choice([2, 3]),
                      4 if hi < 24 else 8, 1e-3, 10, rng.choice([0, 5, 12, 16]), rng.randint(1, 8),
                      rng.randrange(1000))
    mode = rng.choice(["fp64", "mixed", "mixed", "complex"])
    if rng.random() < 0.25:                    # 2-D
        nx = _log_int(rng, 24, 256 if kind == "apply" else 96)
        ny = max(16, int(nx * rng.uniform(0.6, 1.3)))
        return _single(None, kind, "%dx%d" % (nx, ny), 2, rng.choice([2, 4, 8]), "ilu0", 0.0, 0, rng.choice([0, 4, 8]),
                       "fp64" if mode == "complex" else mode, beta=round(rng.uniform(0.0, 0.5), 3),
                       shift=0.05 if mode == "complex" else 0.0, restart=rng.choice([30, 50]))
    side = _log_int(rng, 12, 80 if kind == "apply" else 56 if mode != "complex" else 36)
    dims = [max(9, int(round(side * rng.uniform(0.75, 1.25)))) for _ in range(3)]
    n = dims[0] * dims[1] * dims[2]
    p = 64 if n > 60000 else rng.choice([8, 16]) if n > 8000 else 4
    nlev = rng.choice([3, 4]) if n > 8000 else rng.choice([2, 3])
    tau, lfil = rng.choice([(1e-3, 10), (1e-3, 10), (1e-2, 5)])
    return _single(None, kind, "x".join(map(str, dims)), nlev, p, "ilut", tau, lfil,
                   rng.choice([0, 5, 16, 32] if n > 8000 else [0, 5]), "fp64" if mode == "complex" else mode,
                   beta=round(rng.uniform(0.0, 0.5), 3), local_from=rng.choice([-1, 1]),
                   shift=0.05 if mode == "complex" else 0.0, nrhs=rng.choice([1, 1, 2]),
                   restart=rng.choice([40, 50, 60]))


# ---- problems ---------------------------------------------------------------------------
def _dims(case):
    return tuple(int(t) for t in case["dims"].split("x"))


@functools.lru_cache(maxsize=4)
def _problem(dims, beta, sigma, nlev, p, local_from):
    A, xyz = gi.grid_operator(dims, beta=beta, sigma=sigma)
    return A, partition_geometric(A, xyz, nlev, p, local_from=None if local_from < 0 else local_from)


def _systems(case):
    """(dims, beta) of every system of a batch (the workload's own draw of sides and convection)."""
    return gi.batch_systems(count=case["count"], seed=case["sysseed"], lo=case["lo"], hi=case["hi"])


@functools.lru_cache(maxsize=2)
def _batch_problem(count, lo, hi, sysseed, nlev, p):
    As, parts = [], []
    for dims, beta in gi.batch_systems(count=count, seed=sysseed, lo=lo, hi=hi):
        A, xyz = gi.grid_operator(dims, beta=beta)
        As.append(A)
        parts.append(partition_geometric(A, xyz, nlev, p))
    return As, parts


def _is_batch(case):
    return case["kind"].startswith("batch")


def _of(case):
    if _is_batch(case):
        return _batch_problem(case["count"], case["lo"], case["hi"], case["sysseed"], case["nlev"], case["p"])
    return _problem(_dims(case), case["beta"], case["sigma"], case["nlev"], case["p"], case["local_from"])


def _rows(case):
    if _is_batch(case):
        return sum(int(np.prod(d)) for d, _ in _systems(case))
    return int(np.prod(_dims(case)))


def _rhs(case, seed):
    """Host right-hand sides, uniform in [-1, 1) (both parts of a complex one): (nrhs, n), or the flat batch vector."""
    rng = np.random.default_rng(seed)
    n, nrhs = _rows(case), case["nrhs"]
    if _is_batch(case):
        return rng.uniform(-1.0, 1.0, n * nrhs)
    b = rng.uniform(-1.0, 1.0, (nrhs, n))
    return b + 1j * rng.uniform(-1.0, 1.0, (nrhs, n)) if case["shift"] else b


def prepare(case, seed):
    opts = dict(ilu=case["ilu"], tau=case["tau"], lfil=case["lfil"], rank=case["rank"])
    A, part = _of(case)
    b = torch.from_numpy(_rhs(case, seed)).cuda()
    if _is_batch(case):
        return dict(case=case, handle=GemslrBatch(A, part, **opts), b=b)
    handle = Gemslr(A, part, precision=case["precision"], shift=case["shift"], **opts)
    return dict(case=case, handle=handle, b=b[0] if case["nrhs"] == 1 else b.t())


def run(state):
    case, handle, b = state["case"], state["handle"], state["b"]
    if case["kind"] == "apply":
        return handle.apply(b)
    if case["kind"] == "batch_apply":
        return handle.apply(b, case["nrhs"])
    if case["kind"] == "batch_solve":
        x, info = handle.solve(b, case["nrhs"], restart=case["restart"], rtol=RTOL)
    else:
        x, info = handle.solve(b, restart=case["restart"], rtol=RTOL)
    return {"x": x, "iters": np.array([i["iters"] for i in info]),
            "converged": np.array([i["converged"] for i in info], dtype=np.int64)}


# ---- what a pass cannot do without -----------------------------------------------------
def _apply_work(n, tails, rank, per_row, sv, sw):
    """Bytes and flops of one application to one vector: every factor, coupling block and W read once;
    L and U of a Schur level act twice (down and up), the last level's once."""
    nnz = per_row * n
    last = tails[-1] if tails else n
    couple = 2 * 2 * (tails[0] if tails else 0)          # E and F: about two entries per interface row each
    w = sum(t * min(rank, t) for t in tails)
    vec = 2 * n * (16 if sv == 16 else 8)
    cx = 4 if sv == 16 else 1
    return (nnz + couple) * (sv + 4) + w * sw + vec, cx * (2 * per_row * (2 * n - last) + 2 * couple + 4 * w)


def work(case):
    if _is_batch(case):
        As, parts = _of(case)
        prob = [(A, p, d) for A, p, (d, _) in zip(As, parts, _systems(case))]
        sv, sw = 4, 2
    else:
        A, part = _of(case)
        prob = [(A, part, _dims(case))]
        sv, sw = (16, 16) if case["shift"] else (8, 8) if case["precision"] == "fp64" else (4, 2)
    nb = nf = 0.0
    vs = 16 if sv == 16 else 8
    for A, part, dims in prob:
        tails = [int(A.n - t) for t in part["level_ptr"][1:-1]]
        # ILUT keeps lfil entries in L and in U of almost every row; ILU(0) keeps the stencil
        per_row = 2 * case["lfil"] + 1 if case["ilu"] == "ilut" else 2 * len(dims) + 1
        fb, ff = _apply_work(A.n, tails, case["rank"], per_row, sv, sw)
        if case["kind"].endswith("apply"):
            vec = 2 * A.n * vs
            nb += fb + (case["nrhs"] - 1) * vec
            nf += ff * case["nrhs"]
            continue
        # a solve: about this many steps, each one application, one product with A, and the basis
        # read twice (coefficients, subtraction) in two Gram-Schmidt passes of arithmetic
        side = A.n ** (1.0 / len(dims))
        its = max(4.0, 1.1 * side if len(dims) == 2 else 42.0 * (side / 64.0) ** 0.8)
        cols = min(its, case["restart"]) / 2.0
        shared = fb - 2 * A.n * vs + A.nnz * 12            # read once for all right-hand sides of a step
        per_rhs = 2 * cols * A.n * vs + 4 * A.n * vs
        many = 1 if _is_batch(case) else case["nrhs"]      # a single handle solves them one after another
        nb += its * (shared * many + per_rhs * case["nrhs"])
        nf += its * case["nrhs"] * (ff + 2 * A.nnz + (4 if sv == 16 else 1) * 8 * cols * A.n)
    return {"bytes": float(nb), "flops": float(nf)}


# ---- the exact solution of a solve -------------------------------------------------------
def _axis(d, beta):
    """Eigenvectors, their inverse and eigenvalues of one axis' tridiagonal Toeplitz operator (d unknowns)."""
    h = 1.0 / (d + 1)
    lo, up = -1.0 / h ** 2 - beta / (2 * h), -1.0 / h ** 2 + beta / (2 * h)
    i = np.arange(1, d + 1)
    S = math.sqrt(2.0 / (d + 1)) * np.sin(np.outer(i, i) * (math.pi / (d + 1)))
    lam = 2.0 / h ** 2 - 2.0 * math.sqrt(lo * up) * np.cos(i * (math.pi / (d + 1)))
    scale = (lo / up) ** (0.5 * np.arange(d))
    return scale[:, None] * S, S / scale[None, :], lam


def _solve_exact(dims, beta, sigma, b):
    """A^{-1} b for the separable grid operator (b: (nrhs, n), first axis fastest), by its eigenvectors."""
    axes = [_axis(d, beta) for d in dims]
    nd = len(dims)
    t = b.reshape((b.shape[0],) + tuple(reversed(dims)))
    lam = np.zeros(tuple(reversed(dims)))
    for a, (_, _, l) in enumerate(axes):
        lam = lam + l.reshape([-1 if nd - 1 - q == a else 1 for q in range(nd)])
    lam = lam - sigma * (dims[0] + 1) ** 2
    for pick in (1, 0):                         # into the eigenbasis, divide, back
        for a in range(nd):
            M, ax = axes[a][pick], nd - a
            t = np.moveaxis(np.tensordot(t, M, axes=([ax], [1])), -1, ax)
        if pick == 1:
            t = t / lam
    return np.ascontiguousarray(t).reshape(b.shape[0], -1)


def exact(case, seed):
    """The solution of a solve; an application has none (its factors are the library's)."""
    if not case["kind"].endswith("solve"):
        return None
    b = _rhs(case, seed)
    if not _is_batch(case):
        x = _solve_exact(_dims(case), case["beta"], case["sigma"], b)
        return {"x": torch.from_numpy(x[0]) if case["nrhs"] == 1 else torch.from_numpy(x).t(), "iters": None,
                "converged": None}
    out, o = [], 0
    for dims, beta in _systems(case):
        k = int(np.prod(dims)) * case["nrhs"]
        out.append(_solve_exact(dims, beta, 0.0, b[o:o + k].reshape(case["nrhs"], -1)).ravel())
        o += k
    return {"x": torch.from_numpy(np.concatenate(out)), "iters": None, "converged": None}
