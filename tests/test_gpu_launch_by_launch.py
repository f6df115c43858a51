"""FGMRES launch by launch, which restarts above 60 take on every matrix: the fused Arnoldi step
over its work splits (1, 2, 4 and 8 rows a thread in registers, the sweeping kernel) and the lockstep
blocks with columns that end early.  A cycle that stops on its own residual estimate must have
reached the true residual too: with a wrong dot product, norm or rotation the estimate and the
residual part and the solve needs another cycle."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from paper_2009_06954_gb300.binding import kernel_launches
from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from workloads import dissipative_hamiltonian_3d

pytestmark = pytest.mark.gpu


def _launches(call):
    l0 = kernel_launches()
    out = call()
    return out, kernel_launches() - l0


@pytest.mark.parametrize("side", [3, 7, 34, 43, 54, 68])
def test_one_cycle_reaches_the_residual(pkg, side):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=side, seed=side, with_rhs=False)[0]
    x = np.random.default_rng(side).standard_normal(A.shape[0])
    # two inner steps: the preconditioner is weak, so the cycle passes six vectors
    s = pkg.Solver(A, precision="fp64", outer="fgmres", inner_tol=1e-30, inner_maxit=2, setup_tol=1e-8, outer_tol=1e-10,
                   lls_tol=1e-4, restart=62)
    (xg, st), launches = _launches(lambda: s.solve(A @ x))
    assert launches >= 3 * st["outer_its"]   # mrs, operator and Arnoldi launches of each step
    assert st["status"] == 0 and st["cycles"] == 1 and st["outer_its"] >= (7 if side > 3 else 2), st
    # ||A^-1|| ||A|| of this family is below 4
    assert np.linalg.norm(xg - x) <= 4e-10 * np.linalg.norm(x)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_lockstep_blocks_match_direct(pkg, precision):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=16, seed=9, with_rhs=False)[0]
    n = A.shape[0]
    B = np.random.default_rng(61).standard_normal((n, 11))   # one block of 8 and one of 3
    B[:, 4] = 0.0
    B[:, 7] = 3.0 * B[:, 1]
    B[:, 9] = A @ np.ones(n)                                 # smooth: another number of steps
    s = pkg.Solver(A, precision=precision, outer="fgmres", inner_tol=1e-6 if precision == "mixed" else 1e-10,
                   rhs_block=True, restart=62)
    (X, st), launches = _launches(lambda: s.solve(B))
    assert st["status"] == 0 and st["inner_solves"] > 0 and launches >= 3 * st["outer_its"]
    assert np.all(X[:, 4] == 0)
    Xd = spla.splu(A.tocsc()).solve(B)
    for c in range(B.shape[1]):
        if c == 4:
            continue
        assert np.linalg.norm(B[:, c] - A @ X[:, c]) <= 1e-8 * np.linalg.norm(B[:, c])
        np.testing.assert_allclose(X[:, c], Xd[:, c], rtol=0, atol=1e-7 * np.abs(Xd[:, c]).max())
    for c in (0, 9):                                         # the same as a call with that column alone
        x1, st1 = s.solve(B[:, c])
        assert st1["status"] == 0 and abs(st1["outer_its"] - st["outer_its"]) <= 3
        np.testing.assert_allclose(X[:, c], x1, rtol=0, atol=1e-7 * np.abs(x1).max())
