"""Where a whole solve takes b from and puts x: column strides as the C interface allows them, in place,
and b at a device address that is not a multiple of 8; every form gives the x of the plain call."""
import ctypes as C

import numpy as np
import pytest

from paper_2009_06954_gb300.binding import Stats
from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from workloads import dissipative_hamiltonian_3d

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[9, 48], ids=["cluster", "grid"])
def system(request, pkg):  # noqa: F811
    A = dissipative_hamiltonian_3d(side=request.param, seed=4, with_rhs=False)[0]
    B = np.asfortranarray(A @ np.random.default_rng(2).standard_normal((A.shape[0], 2)))
    s = pkg.Solver(A, precision="mixed", outer="fgmres", inner_tol=1e-3, outer_tol=1e-9)
    return s, B, [s.solve(B)[0], s.solve(B[:, 0].copy())[0]]


def _solve(pkg, s, nrhs, b, ldb, x, ldx):  # noqa: F811
    st = Stats()
    status = pkg.lib().asss_solve(s._h, nrhs, C.c_void_p(b), ldb, C.c_void_p(x), ldx, C.byref(st))
    assert status == 0, pkg.lib().asss_last_error()


@pytest.mark.parametrize("ldb,ldx", [(5, 0), (0, 3)])
def test_host_column_strides(pkg, system, ldb, ldx):  # noqa: F811
    s, B, (X, _) = system
    n = B.shape[0]
    b, x = np.empty(2 * (n + ldb)), np.empty(2 * (n + ldx))
    for c in range(2):
        b[c * (n + ldb):c * (n + ldb) + n] = B[:, c]
    _solve(pkg, s, 2, b.ctypes.data, n + ldb, x.ctypes.data, n + ldx)
    for c in range(2):
        np.testing.assert_array_equal(x[c * (n + ldx):c * (n + ldx) + n], X[:, c])


@pytest.mark.parametrize("pad", [0, 3])
def test_device_column_strides_and_overlap(pkg, system, pad):  # noqa: F811
    import torch
    s, B, (X, _) = system
    n = B.shape[0]
    b = torch.zeros(2 * (n + pad), dtype=torch.float64, device="cuda")
    for c in range(2):
        b[c * (n + pad):c * (n + pad) + n] = torch.tensor(B[:, c], device="cuda")
    torch.cuda.synchronize()
    _solve(pkg, s, 2, b.data_ptr(), n + pad, b.data_ptr(), n + pad)   # in place
    got = b.cpu().numpy()
    for c in range(2):
        np.testing.assert_array_equal(got[c * (n + pad):c * (n + pad) + n], X[:, c])


@pytest.mark.parametrize("nrhs", [1, 2])
def test_unaligned_b_on_the_device(pkg, system, nrhs):  # noqa: F811
    import torch
    s, B, want = system
    n = B.shape[0]
    raw = np.zeros(8 * (nrhs * n + 1), dtype=np.uint8)
    raw[4:4 + 8 * nrhs * n] = np.frombuffer(B[:, :nrhs].ravel(order="F").tobytes(), dtype=np.uint8)
    b = torch.tensor(raw, device="cuda")
    x = torch.empty(nrhs * n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    _solve(pkg, s, nrhs, b.data_ptr() + 4, n, x.data_ptr(), n)
    np.testing.assert_array_equal(x.cpu().numpy(), want[0 if nrhs == 2 else 1].ravel(order="F"))
