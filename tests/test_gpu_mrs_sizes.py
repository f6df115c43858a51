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
