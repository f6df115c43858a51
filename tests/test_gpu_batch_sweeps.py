"""The batched kernel's Gram-Schmidt at the edges of its sweeps: up to six Krylov vectors go
through one fused sweep, more through chunks of six; restarts below, at and above that, with an
inner solve so loose that the cycles are full."""
import numpy as np
import pytest

from test_gpu_batch import _check_columns, pkg  # noqa: F401  (the fixture)
from workloads import batched_dissipative_hamiltonian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restart", [1, 5, 6, 7, 13, 30])
def test_long_cycles_meet_the_tolerance(pkg, restart):  # noqa: F811
    batch = batched_dissipative_hamiltonian(count=3, side_lo=3, side_hi=9, nrhs=2, seed=5)
    As, Bs = [A for A, _ in batch], [B for _, B in batch]
    bs = pkg.BatchSolver(As, inner_tol=0.2, restart=restart)
    x, st = bs.solve(bs.pack(Bs), nrhs=2)
    assert st["status"] == 0 and st["relres"] <= 1e-8
    assert st["outer_its"] > 7
    _check_columns(batch, bs.unpack(x, 2), Bs)
    for (A, _), X, B in zip(batch, bs.unpack(x, 2), Bs):
        # residual 1e-8 through a condition number far below 100
        xs = np.linalg.solve(A.toarray(), B)
        assert np.linalg.norm(X - xs) <= 1e-6 * np.linalg.norm(xs)
    bs.close()
