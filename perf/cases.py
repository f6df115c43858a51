"""Performance cases of the solve path, each one call that a user's program makes.

Every case goes through the public Python entry points (``Solver``, ``BatchSolver``)
with option sets that the benchmark, the named workload configurations or the tests
use.  ``prepare`` builds what a program holds before the call (matrix, set-up handle,
right-hand side on the GPU or the host); ``run`` is the call.

Right-hand sides are b = A x with a drawn x ~ N(0, 1), so the value in 64 bits of a
solve is x itself (the matrices' condition numbers are below 10^4, so the rounding of b moves
it by less than 10^-12).
"""
import math

import numpy as np
import torch

import paper_2009_06954_gb300 as pkg
import workloads

# Option sets.  MIXED: FP32 inner mrs inside FP64 flexible GMRES, the benchmark's choice;
# FP64: the same method without 32-bit arithmetic (the benchmark's comparison leg);
# PAPER: the library's defaults, which are the paper's (FP64, TFQMR, inner tolerance
# 1e-10), at an outer tolerance where the iterates of TFQMR have settled.
MIXED = dict(precision="mixed", outer="fgmres", inner_tol=1e-3, outer_tol=1e-8, k=20)
FP64 = dict(precision="fp64", outer="fgmres", inner_tol=1e-3, outer_tol=1e-8, k=20)
PAPER = dict(precision="fp64", outer="tfqmr", inner_tol=1e-10, outer_tol=1e-11, k=20)
BATCHED = dict(inner_tol=1e-3, outer_tol=1e-8, k=20, restart=24)
GENERAL = dict(precision="mixed", outer="fgmres", inner_tol=1e-6, outer_tol=1e-8, k=20, lls_maxit=400)


def listed():
    return [
        # the smallest system of the batched workload as a call of its own: latency, launches
        {"name": "solve_dh10", "kind": "solve", "side": 10, "host": False},
        # an ordinary time step of a program that keeps its vectors on the host (odd grid)
        {"name": "solve_dh47_host", "kind": "solve", "side": 47, "host": True},
        # the headline: one implicit-Euler step of the 100^3 dissipative-Hamiltonian system
        {"name": "solve_dh100", "kind": "solve", "side": 100, "host": False},
        # the same path without 32-bit arithmetic
        {"name": "solve_dh64_fp64", "kind": "solve_fp64", "side": 64},
        # the paper's own setting at the size of its test matrices (n = 822..5000), library
        # defaults: FP64, TFQMR, long inner solves
        {"name": "solve_cd47_tfqmr", "kind": "tfqmr", "m": 47},
        # several right-hand sides of one system, solved in lockstep (App. B)
        {"name": "solve_dh48_rhs8", "kind": "block", "side": 48, "nrhs": 8},
        # backward pass: adjoint solve and the gradient of A's values
        {"name": "adjoint_dh64", "kind": "adjoint", "side": 64},
        # many small systems of uneven size x many right-hand sides in one launch
        {"name": "batched_32x32", "kind": "batched", "count": 32, "side_lo": 10, "side_hi": 32, "nrhs": 32},
        # a general pattern with heavy-tailed rows (SELL storage)
        {"name": "solve_general_20011", "kind": "general", "n": 20011},
        # the incomplete L D L^T factor of the paper's ~ildl(0): triangular solves inside mrs
        {"name": "solve_dh24_ildl0", "kind": "ildl0", "side": 24},
        # everything that does not depend on b, paid for each new matrix
        {"name": "setup_dh32", "kind": "setup", "side": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve_fp64", "tfqmr", "block", "adjoint", "batched", "general", "ildl0",
                       "setup"])
    if kind == "solve":   # the number of unknowns over its logarithm: 10^3..100^3
        return {"kind": kind, "side": _log_int(rng, 10, 99), "host": rng.random() < 0.5}
    if kind == "solve_fp64":
        return {"kind": kind, "side": _log_int(rng, 10, 63)}
    if kind == "tfqmr":
        return {"kind": kind, "m": rng.randint(24, 46)}
    if kind == "block":
        return {"kind": kind, "side": _log_int(rng, 10, 47), "nrhs": rng.randint(2, 8)}
    if kind == "adjoint":
        return {"kind": kind, "side": _log_int(rng, 10, 63)}
    if kind == "batched":
        lo = rng.randint(10, 14)
        return {"kind": kind, "count": rng.randint(4, 32), "side_lo": lo, "side_hi": lo + rng.randint(2, 16),
                "nrhs": _log_int(rng, 1, 32)}
    if kind == "general":
        return {"kind": kind, "n": _log_int(rng, 2000, 20000)}
    if kind == "ildl0":
        return {"kind": kind, "side": rng.randint(10, 23)}
    return {"kind": kind, "side": rng.randint(10, 31)}


def _batch_sides(case):
    # uneven sizes over the whole range, in a mixed order that the case alone fixes
    lo, hi = case["side_lo"], case["side_hi"]
    sides = np.random.default_rng([lo, hi, case["count"]]).integers(lo, hi + 1, size=case["count"])
    sides[0] = hi
    return [int(s) for s in sides]


def _matrix(case, seed):
    kind = case["kind"]
    if kind == "tfqmr":
        return workloads.convection_diffusion_2d(m=case["m"], seed=seed)[0]
    if kind == "general":   # every row dominant: the rows for which the method converges
        return workloads.random_powerlaw(n=case["n"], band=1000, dom_frac=1.0, seed=seed)[0]
    return workloads.dissipative_hamiltonian_3d(side=case["side"], seed=seed, with_rhs=False)[0]


def _unknowns(case):
    if case["kind"] == "tfqmr":
        return case["m"] ** 2
    if case["kind"] == "general":
        return case["n"]
    return case["side"] ** 3


def _x(n, nrhs, seed, what=0):
    return np.random.default_rng([seed, 11, what]).standard_normal((nrhs, n))


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        mats, rhs = [], []
        for m, s in enumerate(_batch_sides(case)):
            A = workloads.dissipative_hamiltonian_3d(side=s, seed=1000 * seed + m, with_rhs=False)[0]
            mats.append(A)
            rhs += [A @ v for v in _x(A.shape[0], case["nrhs"], seed, m)]
        return {"kind": kind, "solver": pkg.BatchSolver(mats, **BATCHED), "b": _cuda(np.concatenate(rhs)),
                "nrhs": case["nrhs"]}
    A = _matrix(case, seed)
    n = A.shape[0]
    if kind == "setup":
        return {"kind": kind, "A": A}
    opts = {"solve": MIXED, "solve_fp64": FP64, "tfqmr": PAPER, "block": dict(MIXED, rhs_block=True),
            "adjoint": MIXED, "general": GENERAL, "ildl0": dict(MIXED, factor="ildl0")}[kind]
    state = {"kind": kind, "solver": pkg.Solver(A, **opts)}
    if kind == "block":
        B = np.stack([A @ v for v in _x(n, case["nrhs"], seed)])
        state["b"] = _cuda(B).T   # n x nrhs, column-major
    elif kind == "adjoint":
        state["g"] = _cuda(A.T @ _x(n, 1, seed)[0])
        state["x"] = _cuda(_x(n, 1, seed, 1)[0])
    else:
        b = A @ _x(n, 1, seed)[0]
        state["b"] = b if case.get("host") else _cuda(b)
    return state


def run(state):
    kind = state["kind"]
    if kind == "setup":
        s = pkg.Solver(state["A"], **MIXED)
        out = s.export(state["A"].nnz)
        s.close()
        return out
    s = state["solver"]
    if kind == "batched":
        return s.solve(state["b"], nrhs=state["nrhs"])[0]
    if kind == "adjoint":
        lam, dA, _ = s.solve_adjoint(state["g"], x=state["x"])
        return {"lam": lam, "dA": dA}
    return s.solve(state["b"])[0]


def _stencil(side):
    """Rows and columns of the 7-point pattern, in CSR order."""
    i = np.arange(side ** 3)
    c = [i % side, i // side % side, i // side ** 2]
    cols, ok = [], []
    for a, d in ((2, -1), (1, -1), (0, -1), (0, 0), (0, 1), (1, 1), (2, 1)):
        cols.append(i + d * side ** a)
        ok.append((c[a] + d >= 0) & (c[a] + d < side))
    ok = np.stack(ok, 1)
    return np.repeat(i, ok.sum(1)), np.stack(cols, 1)[ok]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batched":
        return np.concatenate([_x(s ** 3, case["nrhs"], seed, m).ravel()
                               for m, s in enumerate(_batch_sides(case))])
    if kind == "setup":
        # the scalings are row and column maxima; the fit and what follows from it have
        # no closed form
        A = _matrix(case, seed)
        n = A.shape[0]
        rows = np.repeat(np.arange(n), np.diff(A.indptr))
        dr, dc = np.zeros(n), np.zeros(n)
        np.maximum.at(dr, rows, np.abs(A.data))
        dr = 1.0 / dr
        np.maximum.at(dc, A.indices, np.abs(dr[rows] * A.data))
        return {"dr": dr, "dc": 1.0 / dc, "w": None, "d": None, "s_val": None, "Q": None, "alpha": None,
                "neg": None}
    n = _unknowns(case)
    if kind == "block":
        return _x(n, case["nrhs"], seed).T
    if kind == "adjoint":
        lam, x = _x(n, 1, seed)[0], _x(n, 1, seed, 1)[0]
        rows, cols = _stencil(case["side"])
        return {"lam": lam, "dA": -lam[rows] * x[cols]}
    return _x(n, 1, seed)[0]


def work(case):
    """Bytes of the plan and of b read once and x written once; FP operations of one
    application of each of its parts."""
    kind = case["kind"]
    if kind == "batched":
        mean = sum(s ** 3 for s in _batch_sides(case)) / case["count"]
        one = work({"kind": "solve", "side": round(mean ** (1 / 3))})
        vec = 16 * mean * case["nrhs"]
        return {"bytes": case["count"] * (one["bytes"] - 16 * mean + vec),
                "flops": case["count"] * case["nrhs"] * one["flops"]}
    n = _unknowns(case)
    per_row = {"tfqmr": 5, "general": 16}.get(kind, 7)   # entries of A a row
    nnz = per_row * n
    # J~ stands on the pattern of A S + (A S)^T, of which one triangle is needed: stencils
    # have 12 (3D) or 6 (2D) positive offsets there, the general rows about 300 entries above
    # the diagonal, each with its column
    jt = {"tfqmr": 6, "general": 300}.get(kind, 12) * n
    fp = 8 if kind in ("tfqmr", "solve_fp64") else 4
    entry = fp + (4 if kind == "general" else 0)
    plan = 2 * 12 * nnz + jt * entry + 2 * 20 * fp * n   # A and S, J~, Q_k, the low-rank correction
    if kind == "setup":
        return {"bytes": 2 * 12 * nnz + 8 * (4 + 20) * n, "flops": 2 * per_row * nnz + 20 * 4 * jt}
    nrhs = case.get("nrhs", 1)
    out = 16 * n * nrhs + (8 * n + 8 * nnz if kind == "adjoint" else 0)
    return {"bytes": plan + out, "flops": nrhs * (4 * nnz + 4 * jt + 6 * 20 * n)}
