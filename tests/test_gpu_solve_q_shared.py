"""Grid-scope solves that keep Q_k in shared memory, against the launch-by-launch path: the
smallest systems of that path, ragged last slices, every width class, both block sizes (up to
768 rows a block and above), and the last sizes that fit and the first that do not (32 columns: about
250 000 rows on 152 SMs)."""
import numpy as np
import pytest

from test_gpu_parity import pkg  # noqa: F401  (the fixture)
from test_gpu_solve_cluster import OPTS, SAME, banded, both, close
from workloads import pattern_diagonal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(14001, 1), (14016, 8), (15999, 11), (20033, 16), (31337, 20), (40000, 23), (116736, 4),
                                 (116737, 4), (240001, 32), (262145, 32)])
def test_matches(pkg, monkeypatch, n, k):  # noqa: F811
    A = banded(n, (-77, -9, -2, 3, 40), 6).tolil()
    A[3, 3] = -A[3, 3]
    A = A.tocsr()
    s = pkg.Solver(A, s_pattern=pattern_diagonal(n), s_values=np.ones(n), lls_maxit=0, k=k, **OPTS["mixed"])
    assert s.setup_stats["r"] == 1
    rng = np.random.default_rng(7)
    b, g = rng.standard_normal(n), rng.standard_normal(n)
    (xa, sa), (xb, sb) = both(monkeypatch, lambda: s.solve(b))
    close(xa, xb)
    assert [sa[q] for q in SAME] == [sb[q] for q in SAME] and sa["status"] == 0
    (la, _, _), (lb, _, _) = both(monkeypatch, lambda: s.solve_adjoint(g))
    close(la, lb)
