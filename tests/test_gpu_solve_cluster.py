"""Cluster- and grid-scope solves against the launch-by-launch path (which ASSS_TRACE asks for) on every
form that takes them: both inner precisions, forward and adjoint, one to seventeen columns
(chunks of sixteen), fewer rows than a cluster has CTAs, a row permutation, matrices without a
diagonal copy, negative pivots, and right-hand sides and limits that end a solve early.  Same
method and stopping rules, other summation orders."""
import numpy as np
import pytest
import scipy.sparse as sp

from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from workloads import dissipative_hamiltonian_3d, pattern_diagonal

pytestmark = pytest.mark.gpu

OPTS = {"mixed": dict(precision="mixed", outer="fgmres", inner_tol=1e-3, outer_tol=1e-10),
        "fp64": dict(precision="fp64", outer="fgmres", inner_tol=1e-3, setup_tol=1e-10, outer_tol=1e-10)}
SAME = ("status", "outer_its", "cycles", "inner_solves", "inner_its_total")


def both(monkeypatch, call):
    monkeypatch.delenv("ASSS_TRACE", raising=False)
    a = call()
    monkeypatch.setenv("ASSS_TRACE", "1")
    b = call()
    monkeypatch.delenv("ASSS_TRACE")
    return a, b


def close(a, b):
    # both end below the outer tolerance of 1e-10 after the same steps; FP32 roundings of the
    # inner solves move the iterate by far less than that
    np.testing.assert_allclose(a, b, rtol=0, atol=1e-10 * max(np.abs(b).max(), 1e-300))


def banded(n, offsets, seed):
    rng = np.random.default_rng(seed)
    A = sp.diags([0.2 * rng.standard_normal(n - abs(o)) for o in offsets], offsets, shape=(n, n)).tocsr()
    return (A + sp.diags(2.0 + rng.random(n))).tocsr()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("side,nrhs,block", [(2, 1, False), (5, 2, False), (7, 17, False), (11, 3, True), (19, 1, False),
                                             (19, 9, True), (24, 1, False), (31, 2, True)])
def test_columns_match(pkg, monkeypatch, side, nrhs, block, precision):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=side, seed=side, with_rhs=False)[0]
    n = A.shape[0]
    X = np.random.default_rng(side).standard_normal((n, nrhs))
    B = np.asfortranarray(A @ X)
    b = B if nrhs > 1 else B[:, 0].copy()
    s = pkg.Solver(A, rhs_block=block, k=min(20, n), **OPTS[precision])
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(b))
    close(xa, xb)
    assert [sa[k] for k in SAME] == [sb[k] for k in SAME]
    assert np.linalg.norm(xa.reshape(n, -1) - X) <= 1e-9 * np.linalg.norm(X)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("side", [13, 25])
def test_adjoint_matches(pkg, monkeypatch, side, precision):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=side, seed=2, with_rhs=False)[0]
    rng = np.random.default_rng(1)
    g, x = rng.standard_normal(A.shape[0]), rng.standard_normal(A.shape[0])
    s = pkg.Solver(A, **OPTS[precision])
    (la, da, sa), (lb, db, sb) = both(monkeypatch, lambda: s.solve_adjoint(g, x=x))
    close(la, lb)
    close(da, db)
    assert [sa[k] for k in SAME] == [sb[k] for k in SAME]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [1500, 15001])
def test_permutation_and_csr_operators_match(pkg, monkeypatch, n, precision):  # noqa: F811
    offs = [o for o in range(-11, 12) if o and o != 4]      # 22 diagonals: no diagonal copy of Abar
    Ab = banded(n, offs, 3)
    perm = np.random.default_rng(4).permutation(n)
    A = sp.csr_matrix((n, n)).tolil()
    A = Ab[np.argsort(perm)].tocsr()                        # row perm[i] of A is row i of the band
    A.sort_indices()
    s = pkg.Solver(A, row_perm=perm, s_pattern=pattern_diagonal(n), **OPTS[precision])
    rng = np.random.default_rng(5)
    b, g = rng.standard_normal(n), rng.standard_normal(n)
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(b))
    close(xa, xb)
    assert [sa[k] for k in SAME] == [sb[k] for k in SAME] and sa["status"] == 0
    (la, _, _), (lb, _, _) = both(monkeypatch, lambda: s.solve_adjoint(g))
    close(la, lb)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,loads", [(700, ""), (14001, ""), (14001, "1")])
def test_negative_pivots_match(pkg, monkeypatch, n, loads, precision):  # noqa: F811
    if loads:
        monkeypatch.setenv("ASSS_FORCE_EVICT_FIRST", loads)
    A = banded(n, (-9, -2, 3), 6).tolil()
    for i in (0, 5, 333, n - 1):
        A[i, i] = -A[i, i]
    A = A.tocsr()
    s = pkg.Solver(A, s_pattern=pattern_diagonal(n), s_values=np.ones(n), lls_maxit=0, **OPTS[precision])
    assert s.setup_stats["r"] == 4
    rng = np.random.default_rng(7)
    b, g = rng.standard_normal(n), rng.standard_normal(n)
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(b))
    close(xa, xb)
    assert [sa[k] for k in SAME] == [sb[k] for k in SAME] and sa["status"] == 0
    (la, _, _), (lb, _, _) = both(monkeypatch, lambda: s.solve_adjoint(g))
    close(la, lb)


@pytest.mark.parametrize("side", [9, 24])
@pytest.mark.parametrize("what", ["zero", "nan", "inf", "maxit", "restart", "tol_one", "in_place"])
def test_early_ends_match(pkg, monkeypatch, what, side):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=side, seed=9, with_rhs=False)[0]
    n = A.shape[0]
    # an iterate that a limit cut off carries the FP32 roundings of its inner solves: FP64 there
    opts = dict(OPTS["fp64" if what == "maxit" else "mixed"], inner_maxit=2)
    opts.update({"maxit": dict(outer_maxit=3), "restart": dict(restart=2), "tol_one": dict(outer_tol=1.0)}.get(what, {}))
    b = np.random.default_rng(9).standard_normal(n)
    b = {"zero": 0.0 * b, "nan": np.where(np.arange(n) == 5, np.nan, b), "inf": np.where(np.arange(n) == 5, np.inf, b)
         }.get(what, b)
    s = pkg.Solver(A, **opts)
    if what == "in_place":
        import torch
        c, d = torch.tensor(b, device="cuda"), torch.tensor(b, device="cuda")
        s.solve(c, x=c)
        monkeypatch.setenv("ASSS_TRACE", "1")
        s.solve(d, x=d)
        close(c.cpu().numpy(), d.cpu().numpy())
        return
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(b))
    assert [sa[k] for k in SAME] == [sb[k] for k in SAME], (sa, sb)
    if what in ("nan", "inf"):
        assert sa["status"] == 4
        np.testing.assert_array_equal(xa, xb)
    else:
        close(xa, xb)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("case", ["dh3", "dh11", "dh20", "pairs", "general"])
def test_incomplete_factor_matches(pkg, monkeypatch, case, precision):  # noqa: F811
    """Triangular sweeps in shared memory: fewer rows than CTAs, colours with more rows than a
    CTA has threads, 2x2 pivots with U_r columns of two entries, rows longer than the
    entries fetched ahead."""
    from workloads import random_powerlaw, saddle_pairs
    opts = dict(OPTS[precision], factor="ildl0")
    if case.startswith("dh"):
        A = dissipative_hamiltonian_3d(side=int(case[2:]), seed=4, with_rhs=False)[0]
    elif case == "pairs":
        A = saddle_pairs(300, seed=5, singles=40)
        n = A.shape[0]
        opts.update(factor="ildl0_bk", s_pattern=sp.identity(n, format="csr"), s_values=np.ones(n), lls_maxit=0,
                    inner_tol=1e-8, r_max=256)
    else:
        A = random_powerlaw(n=400, lmin=4, lmax=60, band=50, dom_frac=1.0, seed=6)[0]
        opts.update(s_pattern=pattern_diagonal(400), lls_maxit=50)
    n = A.shape[0]
    s = pkg.Solver(A, k=min(20, n), **opts)
    rng = np.random.default_rng(8)
    X = rng.standard_normal((n, 2))
    B = np.asfortranarray(A @ X)
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(B))
    close(xa, xb)
    assert [sa[k] for k in SAME] == [sb[k] for k in SAME] and sa["status"] == 0
    g = rng.standard_normal(n)
    (la, _, _), (lb, _, _) = both(monkeypatch, lambda: s.solve_adjoint(g))
    close(la, lb)
