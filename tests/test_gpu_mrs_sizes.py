"""The persistent mrs kernel at the edges of its work split: less than one slice, one row
past a slice, past a block's warps, past one slice per SM and past one round of every warp of the
GPU; padded widths whose k + 1 sums take one, two and three warp folds."""
import numpy as np
import pytest

import oracle as O
from test_gpu_parity import banded_skew, pkg  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,fmt", [("fp64", "diag"), ("fp64", "sell"), ("mixed", "diag")])
@pytest.mark.parametrize("n,k", [(9, 0), (31, 3), (33, 8), (257, 31), (4865, 20), (4865, 60), (38945, 20)])
def test_mrs_iterate_at_split_edges(pkg, n, k, precision, fmt):  # noqa: F811
    J = banded_skew(n, (1, 3) if n < 64 else (1, 3, 17), seed=n + k)
    rng = np.random.default_rng(n)
    b = rng.standard_normal(n)
    Q = alpha = None
    apply = lambda V: J @ V  # noqa: E731
    if k:
        Q, alpha = O.skew_lanczos(J, rng.standard_normal(n), k)
        Sk = O.lanczos_tridiagonal(alpha)
        apply = lambda V: J @ V - Q @ (Sk @ (Q.T @ V))  # noqa: E731
    xo, its_o, ratio_o, _ = O.mrs(1.0, apply, b, 4, 1e-30)
    x, its, ratio = pkg.mrs(J, b, Q, alpha, tol=1e-30, maxit=4, precision=precision, fmt=fmt)
    assert its == its_o
    # four steps of a recurrence with coefficients of order one: a few hundred roundings
    rtol = 1e-12 if precision == "fp64" else 2e-5
    assert abs(ratio - ratio_o) <= rtol * max(ratio_o, 1.0)
    np.testing.assert_allclose(x, xo, rtol=0, atol=rtol * np.abs(xo).max())


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,q_bf16", [(150, False), (1001, False), (5003, False), (5003, True)])
def test_long_rows_match_sell(pkg, n, q_bf16, precision, monkeypatch):  # noqa: F811
    """J~ with long rows (one of them full, one empty but for its diagonal) through the
    row-stream pass against the SELL pass of the same set-up: the same products in another
    order.  Fewer rows than SMs, a row longer than a warp's share, evict-first loads."""
    from workloads import random_powerlaw
    if q_bf16 and precision == "fp64":
        pytest.skip("BF16 Q belongs to the FP32 solve")
    A = random_powerlaw(n=n, lmin=4, lmean=16.0, lmax=min(512, n // 2), band=n // 4, dom_frac=1.0, seed=n)[0].tolil()
    A[7, :] = 0.01
    A[7, 7] = 0.02 * n
    A[n - 3, :] = 0.0
    A[:, n - 3] = 0.0
    A[n - 3, n - 3] = 1.0
    A = A.tocsr()
    if q_bf16:
        monkeypatch.setenv("ASSS_FORCE_EVICT_FIRST", "1")
    rng = np.random.default_rng(n)
    u = rng.standard_normal(n)
    opts = dict(precision=precision, outer="fgmres", inner_tol=1e-11 if precision == "fp64" else 1e-5, setup_tol=1e-11,
                lls_maxit=40, q_bf16=q_bf16)
    s = pkg.Solver(A, **opts)
    assert s.setup_stats["nnz_pattern"] >= 65 * n
    z, its = s.apply_preconditioner(u)
    zt, _ = s.apply_preconditioner(u, transpose=True)
    s2 = pkg.Solver(A, inner_format="sell", **opts)
    z2, its2 = s2.apply_preconditioner(u)
    z2t, _ = s2.apply_preconditioner(u, transpose=True)
    # both stop at the same tolerance, so they may differ by it
    tol = 1e-9 if precision == "fp64" else 1e-4
    assert abs(its - its2) <= 1
    np.testing.assert_allclose(z, z2, rtol=0, atol=tol * np.abs(z2).max())
    np.testing.assert_allclose(zt, z2t, rtol=0, atol=tol * np.abs(z2t).max())
