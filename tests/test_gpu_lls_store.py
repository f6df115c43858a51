"""Which form the least-squares fit takes: B and B^T stored (one launch for the whole iteration) or
applied matrix-free (about eight launches an iteration), by the memory that the stored form
needs with its padding; and the stored form of very uneven rows, whose pairs are sorted."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from paper_2009_06954_gb300.binding import kernel_launches
from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from workloads import pattern_of

pytestmark = pytest.mark.gpu


def _uneven(kind, n, seed=3):
    """Columns of very different lengths: an arrow, a few long columns, power-law columns."""
    rng = np.random.default_rng(seed)
    A = sp.lil_matrix((n, n))
    if kind == "arrow":
        A[0, :] = 0.3 * rng.standard_normal(n) / np.sqrt(n)
        A[:, 0] = 0.3 * rng.standard_normal((n, 1)) / np.sqrt(n)
    elif kind == "columns":      # no entry of a long column has its mirror
        for j in range(0, n, max(n // 5, 1)):
            rows = rng.choice(n, size=n // 2, replace=False)
            A[rows, j] = 0.3 * rng.standard_normal((rows.size, 1)) / np.sqrt(n)
    else:
        for j in range(n):
            rows = rng.choice(n, size=min(n, int(3 / (rng.random() + 0.02))), replace=False)
            A[rows, j] = 0.2 * rng.standard_normal((rows.size, 1)) / np.sqrt(rows.size)
    A = (A + sp.diags(2.0 + rng.random(n))).tocsr()
    A.sort_indices()
    return A


def _fit(pkg, A, gamma=0.5):  # noqa: F811
    Sp = pattern_of(A)
    Abar = sp.csr_matrix(O.equilibrate(A)[0])
    Abar.sort_indices()
    sg, st = pkg.skew_symmetrizer(Abar, Sp, gamma=gamma)
    B, v, (rows, cols) = O.lls_system(Abar, Sp, gamma)
    s = np.asarray(sp.csr_matrix((sg, Sp.indices, Sp.indptr), shape=Sp.shape)[rows, cols]).ravel()
    grad = np.linalg.norm(B.T @ (v - B @ s)) / np.linalg.norm(B.T @ v)
    # the stopping rule is 1e-13 of the start's gradient
    assert st["lls_relgrad"] <= 1e-13 and grad <= 1e-12, (st["lls_relgrad"], grad)
    return sg


@pytest.mark.parametrize("n", [40, 300, 700])
@pytest.mark.parametrize("kind", ["arrow", "columns", "powerlaw"])
def test_both_forms_fit_uneven_columns(pkg, monkeypatch, kind, n):  # noqa: F811
    A = _uneven(kind, n)
    stored = _fit(pkg, A)
    monkeypatch.setenv("ASSS_LLS_STORE_BYTES", "0")
    free = _fit(pkg, A)
    # the same minimiser to the stopping rule, through a normal matrix of condition below 10^4
    np.testing.assert_allclose(stored, free, rtol=0, atol=1e-9 * np.abs(free).max())


def test_the_bound_covers_the_padding(pkg, monkeypatch):  # noqa: F811
    """A bound between what the entries alone take and what they take padded: matrix-free.  In an
    arrow a pair holds a long and a short row, so B^T is stored at nearly twice its entries
    however its pairs are sorted."""
    A = _uneven("arrow", 700)
    Sp = pattern_of(A)
    Abar = sp.csr_matrix(O.equilibrate(A)[0])
    B, _, _ = O.lls_system(Abar, Sp, 0.5)
    entries = 12 * 2 * B.nnz
    # vectors of a slot each: five over the unknowns, two over the constraints
    vectors = 8 * (5 * (Sp.nnz + 31) + 2 * (B.shape[0] + 31))
    runs = {}
    for what, bound in (("none", 0), ("entries", entries + vectors), ("padded", 2.5 * entries + vectors)):
        monkeypatch.setenv("ASSS_LLS_STORE_BYTES", repr(float(bound)))
        launches = []
        for maxit in (2, 7):
            l0 = kernel_launches()
            _, st = pkg.skew_symmetrizer(Abar, Sp, gamma=0.5, lls_tol=0.0, lls_maxit=maxit)
            launches.append(kernel_launches() - l0)
            assert st["lls_its"] == maxit
        runs[what] = (launches[1] - launches[0]) / 5   # launches an iteration
    assert runs["none"] > 4 and runs["entries"] > 4 and runs["padded"] == 0, runs
