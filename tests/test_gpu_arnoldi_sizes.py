"""The fused Arnoldi step over its work splits: 1, 2, 4 and 8 rows a thread in registers and
the sweeping kernel, few vectors and many (shared by several warps, one warp each, more
than the warps of a block).  A cycle that stops on its own residual estimate must have reached
the true residual too: with a wrong dot product, norm or rotation the estimate and the residual
part and the solve needs another cycle."""
import numpy as np
import pytest

from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from workloads import convection_diffusion_2d, dissipative_hamiltonian_3d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [3, 7, 34, 43, 54, 68])
def test_one_cycle_reaches_the_residual_by_rows(pkg, side):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=side, seed=side, with_rhs=False)[0]
    x = np.random.default_rng(side).standard_normal(A.shape[0])
    # two inner steps: the preconditioner is weak, so the cycle passes six vectors
    s = pkg.Solver(A, precision="fp64", outer="fgmres", inner_tol=1e-30, inner_maxit=2, setup_tol=1e-8, outer_tol=1e-10,
                   lls_tol=1e-4, restart=60)
    xg, st = s.solve(A @ x)
    assert st["status"] == 0 and st["cycles"] == 1 and st["outer_its"] >= (7 if side > 3 else 2), st
    # ||A^-1|| ||A|| of this family is below 4
    assert np.linalg.norm(xg - x) <= 4e-10 * np.linalg.norm(x)


@pytest.mark.parametrize("m,inner", [(9, 400), (24, 40), (40, 400)])
def test_one_cycle_reaches_the_residual_by_vectors(pkg, m, inner):  # noqa: F811
    A, b, x = convection_diffusion_2d(m=m)
    s = pkg.Solver(A, precision="fp64", outer="fgmres", inner_tol=1e-10, inner_maxit=inner, outer_tol=1e-9, restart=62)
    xg, st = s.solve(b)
    assert st["status"] == 0 and st["outer_its"] > 6, st
    assert st["cycles"] == (st["outer_its"] + 61) // 62, st
    assert np.linalg.norm(b - A @ xg) <= 1e-9 * np.linalg.norm(b)
