"""The least-squares fit's stored form at the edges of its layout: one row, fewer constraints than
a slice, unknowns without a partner (odd tails), rows longer than the eight entries in
flight and of very different lengths (sorted windows), start values, an iteration limit."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from workloads import pattern_of, random_powerlaw

pytestmark = pytest.mark.gpu


def _matrix(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "powerlaw":
        return random_powerlaw(n=n, lmin=4, lmean=8.0, lmax=n // 3, band=n // 5, dom_frac=1.0, seed=seed)[0]
    A = (sp.eye(n) * 2.0 + 0.2 * sp.random(n, n, density=min(1.0, 3.0 / n), random_state=rng,
                                           data_rvs=rng.standard_normal)).tocsr()
    A.sort_indices()
    return A


@pytest.mark.parametrize("kind,n,pattern", [("random", 1, "A"), ("random", 5, "A"), ("random", 33, "upper"),
                                            ("random", 200, "A"), ("powerlaw", 150, "A"), ("powerlaw", 700, "upper")])
@pytest.mark.parametrize("gamma", [1.0, 0.25])
def test_fit_meets_the_oracles_normal_equations(pkg, kind, n, pattern, gamma):  # noqa: F811
    A = _matrix(kind, n, n)
    # an upper triangular pattern has no pairs at all; A's own has some of both
    Sp = pattern_of(sp.triu(A, format="csr") if pattern == "upper" else A)
    Abar, _, _, _ = O.equilibrate(A)
    Abar = sp.csr_matrix(Abar)
    Abar.sort_indices()
    B, v, (rows, cols) = O.lls_system(Abar, Sp, gamma)
    sg, st = pkg.skew_symmetrizer(Abar, Sp, gamma=gamma)
    S = sp.csr_matrix((sg, Sp.indices, Sp.indptr), shape=Sp.shape)
    s = np.asarray(S[rows, cols]).ravel()
    # the gradient with the oracle's own B and v: the stopping rule is 1e-13 of the start's
    assert st["lls_relgrad"] <= 1e-13
    assert np.linalg.norm(B.T @ (v - B @ s)) <= 1e-12 * np.linalg.norm(B.T @ v)


def test_iteration_limit_and_start_values(pkg):  # noqa: F811
    A = _matrix("powerlaw", 400, 3)
    kw = dict(precision="mixed", outer="fgmres", inner_tol=1e-4)
    s = pkg.Solver(A, lls_maxit=5, **kw)
    assert s.setup_stats["lls_its"] == 5 and s.setup_stats["lls_relgrad"] > 1e-13
    full = pkg.Solver(A, **kw)
    v = full.export(A.nnz)["s_val"]
    again = pkg.Solver(A, s_values=v, **kw)
    assert again.setup_stats["lls_its"] == 0
    np.testing.assert_array_equal(again.export(A.nnz)["s_val"], v)
    part = pkg.Solver(A, s_values=s.export(A.nnz)["s_val"], **kw)
    np.testing.assert_allclose(part.export(A.nnz)["s_val"], v, rtol=0, atol=1e-8 * np.abs(v).max())
