"""Rows over skew diagonals whose loads are issued in groups of twelve: fewer diagonals than a group, one
group, one more than one and two groups, against the oracle; and the whole-solve kernel of large
systems whose Q_k does not fit shared memory, at the smallest size of each narrow width."""
import numpy as np
import pytest

import oracle as O
from test_gpu_parity import banded_skew, pkg  # noqa: F401  (the fixture)
from test_gpu_solve_cluster import SAME, both
from workloads import dissipative_hamiltonian_3d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [0, 5])
@pytest.mark.parametrize("ndiag", [1, 11, 12, 13, 24, 25, 40])
def test_mrs_iterate_by_diagonals(pkg, ndiag, q):  # noqa: F811
    n = 3001
    offs = tuple(int(o) for o in np.cumsum(np.random.default_rng(ndiag).integers(1, 9, size=ndiag)))
    J = banded_skew(n, offs, seed=ndiag)
    J = J * (0.4 / max(1.0, np.sqrt(ndiag)))
    rng = np.random.default_rng(n)
    b = rng.standard_normal(n)
    Q = alpha = None
    apply = lambda V: J @ V  # noqa: E731
    if q:
        Q, alpha = O.skew_lanczos(J, rng.standard_normal(n), q)
        Sk = O.lanczos_tridiagonal(alpha)
        apply = lambda V: J @ V - Q @ (Sk @ (Q.T @ V))  # noqa: E731
    xo, its_o, ratio_o, _ = O.mrs(1.0, apply, b, 4, 1e-30)
    x, its, ratio = pkg.mrs(J, b, Q, alpha, tol=1e-30, maxit=4, precision="mixed", fmt="diag")
    assert its == its_o
    # four steps of a recurrence with coefficients of order one: a few hundred FP32 roundings
    assert abs(ratio - ratio_o) <= 2e-5 * max(ratio_o, 1.0)
    np.testing.assert_allclose(x, xo, rtol=0, atol=2e-5 * np.abs(xo).max())


@pytest.mark.slow
@pytest.mark.parametrize("side,k", [(83, 12), (95, 8), (117, 4)])
def test_large_solves_match_launch_by_launch(pkg, monkeypatch, side, k):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=side, seed=3, with_rhs=False)[0]
    x = np.random.default_rng(side).standard_normal(A.shape[0])
    s = pkg.Solver(A, precision="mixed", outer="fgmres", inner_tol=1e-3, outer_tol=1e-10, lls_tol=1e-3, k=k)
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(A @ x))
    assert [sa[f] for f in SAME] == [sb[f] for f in SAME] and sa["status"] == 0
    # both end below 1e-10 after the same steps; ||A^-1|| ||A|| of this family is below 4
    np.testing.assert_allclose(xa, xb, rtol=0, atol=8e-10 * np.abs(xb).max())
    assert np.linalg.norm(xa - x) <= 4e-10 * np.linalg.norm(x)
