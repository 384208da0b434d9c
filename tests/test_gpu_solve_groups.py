"""Direct solves whose core leaves CTAs over for groups of columns: cores of one block of 64 rows, of a
few, and of enough for the chip, with column counts at the edges of the groups, against a dense FP64
solve on the exported factor.  Bound: backward stable solves of a matrix of condition cond (at most
(lambda + |K~|) / lambda) differ by cond times some n 2^-53."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,tol", [(3, 400, 1e-3), (3, 700, 1e-5), (4, 900, 1e-6), (5, 1200, 1e-5)])
def test_columns_against_dense(d, n, tol):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(n)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), "gaussian", 1.5, tol)
    U, S = f.export()
    A = (U * S) @ U.T
    lam = 0.05 * n
    A[np.diag_indices(n)] += lam
    w = np.linalg.eigvalsh(A)
    assert w[0] > 0
    for c in (64, 1, 2, 7, 8, 9, 16, 17, 31, 63, 65):
        B = np.random.default_rng(7).standard_normal((n, 65))[:, :c]
        X = f.solve(lam, to_dev(B), refine_steps=0).cpu().numpy()
        ref = np.linalg.solve(A, B)
        assert f.device_errors() == 0
        assert np.abs(X - ref).max() <= 4 * n * 2.0 ** -53 * w[-1] / w[0] * np.abs(ref).max(), c


@pytest.mark.parametrize("d,n,tol", [(3, 500, 1e-3), (4, 800, 1e-4)])
@pytest.mark.parametrize("above", [1e-1, 1e-3, 1e-6])
def test_close_to_the_smallest_eigenvalue(d, n, tol, above):
    """lambda just above -lambda_min(K~): lambda I + K~ is nearly singular but positive definite, so the core
    is factored without pivoting.  Backward error: the core C = lambda S^-1 + U^T U is solved to some r
    2^-53 of |C| |z|, and U C^-1 U^T b and b / lambda cancel by at most |b| / (lambda |x|)."""
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(3 * n)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), "cauchy", 0.7, tol)
    U, S = f.export()
    K = (U * S) @ U.T
    w = np.linalg.eigvalsh(K)
    if w[0] >= 0:
        pytest.skip("K~ of these points has full rank and is positive definite")
    lam = -w[0] * (1 + above)
    b = g.standard_normal(n)
    for steps in (0, 1):
        x = f.solve(lam, to_dev(b), refine_steps=steps).cpu().numpy()
        r = lam * x + K @ x - b
        norms = (lam + w[-1]) * np.linalg.norm(x) + np.linalg.norm(b) * (1 + w[-1] / lam)
        assert np.linalg.norm(r) <= 16 * (n + f.rank) * 2.0 ** -53 * norms, steps
