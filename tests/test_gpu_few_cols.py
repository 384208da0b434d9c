"""FP64 products of few columns (streaming kernels) against numpy on the exported factor, at the
edges of their row groups, column steps, row chunks and column counts.

Bound: every entry of U (S (U^T V)) is a sum of n r products of three rounded factors, so in any
order of summation |error| <= 2 (n + r + 4) eps |U| |S| |U|^T |V| entrywise."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,tol", [(3, 1, 1e-6), (3, 7, 1e-6), (3, 9, 1e-8), (4, 255, 1e-3), (3, 2001, 1e-6),
                                     (5, 513, 1e-5), (4, 4099, 1e-4)])
def test_few_columns_match_numpy(d, n, tol):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(100 * d + n)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), "gaussian", 0.7, tol)
    U, S = f.export()
    aU = np.abs(U)
    for c in (1, 2, 3, 4, 5, 65, 67):          # 65 and 67: a group of 64, then one or three columns
        V = g.standard_normal((n, c)) * np.exp(g.uniform(-5, 5, (n, 1)))
        Y = f.matvec(to_dev(V)).cpu().numpy()
        ref = U @ (S[:, None] * (U.T @ V))
        bound = 2 * (n + f.rank + 4) * 2.0 ** -53 * (aU @ (np.abs(S)[:, None] * (aU.T @ np.abs(V))))
        assert np.all(np.abs(Y - ref) <= 2 * bound), c      # twice: numpy's own error


def test_few_columns_cross_and_infinities():
    """Both directions of a cross factor, and a non-finite entry reaches every row it should."""
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(5)
    x, y = g.uniform(-1, 1, (1201, 3)), g.uniform(-1, 1, (333, 3))
    f = hdf.build_cross(to_dev(x), to_dev(y), "cauchy", 1.0, 1e-6)
    U, S = f.export()
    V = f.export_y()
    for c in (1, 3):
        B, W = g.standard_normal((333, c)), g.standard_normal((1201, c))
        for out, ref in ((f.matvec(to_dev(B)), U @ (S[:, None] * (V.T @ B))),
                         (f.matvec_t(to_dev(W)), V @ (S[:, None] * (U.T @ W)))):
            out = out.cpu().numpy()
            assert np.linalg.norm(out - ref) <= 1e-12 * np.linalg.norm(ref)
    b = np.ones(333)
    b[17] = np.nan
    assert np.isnan(f.matvec(to_dev(b)).cpu().numpy()).all()
