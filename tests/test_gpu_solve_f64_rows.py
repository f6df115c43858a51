"""FP64 whole solves on both sides of the line between 256 and 512 threads a block (2048 rows a block on
152 SMs, so 67^3 and 68^3), with and without deflation, against the launch-by-launch path."""
import numpy as np
import pytest

from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from test_gpu_solve_cluster import SAME, both, close
from workloads import dissipative_hamiltonian_3d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,k", [(67, 20), (68, 20), (68, 0), (68, 32)])
def test_both_block_sizes_match(pkg, monkeypatch, side, k):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=side, seed=side, with_rhs=False)[0]
    n = A.shape[0]
    X = np.random.default_rng(side).standard_normal((n, 2))
    B = np.asfortranarray(A @ X)
    s = pkg.Solver(A, precision="fp64", outer="fgmres", inner_tol=1e-3, setup_tol=1e-10, outer_tol=1e-10, lls_tol=1e-4, k=k)
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(B))
    close(xa, xb)
    assert [sa[f] for f in SAME] == [sb[f] for f in SAME] and sa["status"] == 0
    assert np.linalg.norm(xa - X) <= 1e-9 * np.linalg.norm(X)
    g = B[:, 1].copy()
    (la, da, _), (lb, db, _) = both(monkeypatch, lambda: s.solve_adjoint(g, x=X[:, 0].copy()))
    close(la, lb)
    close(da, db)
