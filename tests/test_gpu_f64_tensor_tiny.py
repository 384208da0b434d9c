"""FP64 slice products of columns near the bottom of FP64's range, against extended precision (whose
range goes on below it) on the exported factor.

Bound: that of the slices, 192 x 2^-55 of the largest |a| and |v| of each block of 64, and the FP64 sums,
as for ordinary values; besides, every block sum and every rounding may be off by one unit of the
subnormal numbers, 2^-1074."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu
KB, LD = 64, np.longdouble
EPS, TINY = LD(2.0) ** -53, LD(2.0) ** -1074


def contract(A, V):
    """(A^T V, its error bound) in extended precision."""
    A, V = A.astype(LD), V.astype(LD)
    err = np.zeros((A.shape[1], V.shape[1]), dtype=LD)
    for k0 in range(0, len(A), KB):
        a, v = np.abs(A[k0:k0 + KB]), np.abs(V[k0:k0 + KB])
        err += 192 * LD(2.0) ** -55 * a.max(0)[:, None] * v.max(0)[None, :] + 2 * TINY
    return A.T @ V, err + (len(A) / KB + 3) * EPS * (np.abs(A).T @ np.abs(V)) + TINY


@pytest.mark.parametrize("d,n,tol", [(3, 700, 1e-6), (4, 1025, 1e-3)])
def test_tiny_columns(d, n, tol):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(n)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), "gaussian", 0.8, tol)
    assert f.info.ldu >= 64
    U, S = f.export()
    scales = [0, -940, -957, -960, -985, -1010, -1040, -1065]
    V = g.standard_normal((n, len(scales) + 1))
    for j, s in enumerate(scales):
        V[:, j] = np.ldexp(V[:, j], s)
    V[: n // 2, -1] = np.ldexp(V[: n // 2, -1], -1000)      # tiny blocks, then ordinary ones
    Y = f.matvec(to_dev(V)).cpu().numpy()
    W, e1 = contract(U, V)
    W, e1 = S[:, None] * W, np.abs(S)[:, None] * e1
    e1 += 2 * EPS * np.abs(W) + 2 * TINY
    ref, e2 = contract(np.ascontiguousarray(U.T), W)
    bad = np.abs(Y.astype(LD) - ref) > e2 + np.abs(U) @ e1
    assert not bad.any(), [s for s, b in zip(scales + ["mixed"], bad.any(0)) if b]
    assert all((Y[:, j] != 0).any() for j in range(V.shape[1]))
