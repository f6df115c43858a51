"""More than 32 deflation vectors: the Q_k^T z that the SMW correction reads comes out of one
warp of the mrs kernel, two values a lane above k = 32, on every storage of J~."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from test_gpu_parity import _general_sparse, pkg  # noqa: F401  (the fixture)
from workloads import dissipative_hamiltonian_3d, random_powerlaw

pytestmark = pytest.mark.gpu


def _matrix(case):
    if case == "diagonals":
        return dissipative_hamiltonian_3d(side=13, seed=5, with_rhs=False)[0]
    if case == "diagonals_many":   # more than a slice per SM
        return dissipative_hamiltonian_3d(side=19, seed=5, with_rhs=False)[0]
    if case == "sell":
        return _general_sparse(2001, seed=7)
    return random_powerlaw(n=1500, lmin=4, lmean=16.0, lmax=300, band=300, dom_frac=1.0, seed=3)[0]   # row stream


@pytest.mark.parametrize("precision,q_bf16", [("fp64", False), ("mixed", False), ("mixed", True)])
@pytest.mark.parametrize("case", ["diagonals", "diagonals_many", "sell", "stream"])
@pytest.mark.parametrize("k", [32, 33, 40, 64])
def test_preconditioner_inverts_its_operator(pkg, k, case, precision, q_bf16):  # noqa: F811
    A = _matrix(case)
    s = pkg.Solver(A, precision=precision, inner_tol=1e-10 if precision == "fp64" else 1e-6, setup_tol=1e-12, k=k,
                   q_bf16=q_bf16)
    assert s.setup_stats["k_eff"] == k
    ex = s.export(A.nnz)
    Abar = sp.csr_matrix(O.equilibrate(A)[0])
    S = sp.csr_matrix((ex["s_val"], Abar.indices.copy(), Abar.indptr.copy()), shape=A.shape)
    P = (sp.diags(np.sign(ex["d"])) + O.inner_skew_operator(Abar, S, ex["w"])).tocsr()
    u = np.random.default_rng(11).standard_normal(A.shape[0])
    # the inner tolerance (and Q_k's 8 bits in BF16, which the exact correction does not share)
    # through ||P^-1|| <= 1 and the correction
    bound = 1e-8 if precision == "fp64" else 2e-2 if q_bf16 else 1e-4
    for tr in (False, True):
        # twice: the second call finds what the first left in the correction's buffer
        for _ in range(2):
            z, its = s.apply_preconditioner(u, transpose=tr)
            assert its > 0
            r = ((P.T if tr else P) @ z) - u
            assert np.linalg.norm(r) <= bound * np.linalg.norm(u), (tr, np.linalg.norm(r) / np.linalg.norm(u))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solve_and_adjoint(pkg, precision):  # noqa: F811
    A = _matrix("diagonals")
    rng = np.random.default_rng(1)
    b, g = rng.standard_normal(A.shape[0]), rng.standard_normal(A.shape[0])
    s = pkg.Solver(A, precision=precision, outer="fgmres", inner_tol=1e-8 if precision == "fp64" else 1e-4, outer_tol=1e-10,
                   k=50)
    x, st = s.solve(b)
    assert st["status"] == 0 and np.linalg.norm(b - A @ x) <= 1e-10 * np.linalg.norm(b)
    lam, _, sa = s.solve_adjoint(g)
    assert sa["status"] == 0 and np.linalg.norm(g - A.T @ lam) <= 1e-10 * np.linalg.norm(g)
    # a preconditioner that is applied right to its tolerance leaves the outer method few steps
    ref = pkg.Solver(A, precision=precision, outer="fgmres", inner_tol=1e-8 if precision == "fp64" else 1e-4,
                     outer_tol=1e-10, k=32)
    _, sr = ref.solve(b)
    assert st["outer_its"] <= sr["outer_its"] + 1
