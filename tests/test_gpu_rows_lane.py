"""Rows of narrow FP32 factors (lane-per-point kernel) against the FP64 factor of the same points,
whose rows the two-kernel form writes: same degree, and K~V within the FP32 rounding of the rows.

Bound: an entry of U is a product of d - 1 level and trigonometric factors, each off by a few FP32
roundings of recurrences of length <= L (together below 64 eps32 of the harmonic's bound), times a
radial factor off by a few eps32, so |U S U^T v| differs by at most 256 eps32 |U| |S| |U|^T |v|; the
two factors may drop different eigenpairs at the budget boundary, within tol |K|_F |v|."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,tol", [(3, 1e-2), (3, 1e-4), (4, 1e-3), (5, 1e-3), (6, 1e-2), (7, 1e-2), (8, 1e-1)])
@pytest.mark.parametrize("n", [1, 31, 33, 1025, 60001])
def test_narrow_rows(d, tol, n):
    import torch
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(100 * d + n)
    x = g.standard_normal((n, d))
    x /= np.linalg.norm(x, axis=1).max()
    if n > 40:
        x[7] = 0.0
        x[11, :2] = 0.0                      # x_0 = x_1 = 0: no azimuth
        x[13, 1:] = 0.0                      # on the first axis
    xt = to_dev(x)
    f = hdf.build(xt, "cauchy", 1.0, tol, precision="fp32")
    h = hdf.build(xt, "cauchy", 1.0, tol, precision="fp64")
    assert f.info.p == h.info.p
    V = g.standard_normal((n, 3))
    Y = f.matvec(to_dev(V).float()).double().cpu().numpy()
    U, S = h.export()
    ref = U @ (S[:, None] * (U.T @ V))
    bound = 256 * 2.0 ** -24 * (np.abs(U) @ (np.abs(S)[:, None] * (np.abs(U).T @ np.abs(V))))
    slack = tol * n * np.sqrt(f.info.mu2) * np.linalg.norm(V, axis=0)
    assert np.all(np.linalg.norm(Y - ref, axis=0) <= np.linalg.norm(bound, axis=0) + slack)
    if f.s_k == h.s_k:
        assert np.all(np.linalg.norm(Y - ref, axis=0) <= np.linalg.norm(bound, axis=0))
        A, SA = f.export()
        assert A.shape == U.shape
        # entrywise up to the sign of an eigenvector, where the spectrum separates them: |A| S |A|^T
        assert np.allclose((A.astype(float) ** 2).sum(1), (U ** 2).sum(1), rtol=2e-4, atol=1e-5 * (U ** 2).sum(1).max())
