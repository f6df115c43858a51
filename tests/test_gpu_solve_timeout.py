"""A whole solve whose grid barriers run out: the call says so for one column and for several, every
block still leaves, and the GPU goes on working.  The set-up of these solvers crosses no grid
barrier (least-squares fit matrix-free, no deflation vectors, no negative pivots), so the first
wait is the solve's own."""
import numpy as np
import pytest

from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from workloads import dissipative_hamiltonian_3d

pytestmark = pytest.mark.gpu

TIMEOUT = 8


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_timeout_is_reported_and_a_later_solve_is_right(pkg, monkeypatch, precision):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=47, seed=4, with_rhs=False)[0]   # three columns in grid scope too
    n = A.shape[0]
    X = np.random.default_rng(2).standard_normal((n, 3))
    B = np.asfortranarray(A @ X)
    opts = dict(precision=precision, outer="fgmres", k=0, inner_tol=1e-3, outer_tol=1e-9)
    good = pkg.Solver(A, **opts)
    assert good.setup_stats["r"] == 0
    before = good.solve(B)
    monkeypatch.setenv("ASSS_LLS_STORE_BYTES", "0")
    short = pkg.Solver(A, wait_timeout_ms=1e-6, **opts)
    for b in (B[:, 0].copy(), B, B):
        with pytest.raises(pkg.AsssError) as e:
            short.solve(b)
        assert e.value.status == TIMEOUT
    with pytest.raises(pkg.AsssError) as e:
        short.solve_adjoint(B[:, 0].copy())
    assert e.value.status == TIMEOUT
    after = good.solve(B)
    np.testing.assert_array_equal(before[0], after[0])
    assert after[1]["status"] == 0 and np.linalg.norm(after[0] - X) <= 1e-7 * np.linalg.norm(X)
