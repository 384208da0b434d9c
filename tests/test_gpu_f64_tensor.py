"""FP64 products on the tensor cores (exact integer slices) against extended precision on the
exported factor, at the edges of their tiles, blocks, column groups and exponent rules.

Bound, with blocks of 64 along each contraction: truncating both factors and dropping the lowest
slice products loses at most 3 x 2^-55 of (largest |u|)(largest |v|) of the block per product, and
the block sums are added in FP64: with b blocks
  |error of A^T v| <= sum_blocks 192 2^-55 max|a| max|v| + (b + 2) 2^-53 |A|^T |v|,
applied to U^T V and to U (S W), the first error carried through |U| |S|."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu
KB = 64


def contract(A, V):
    """(A^T V in extended precision, its error bound) for A (k, m), V (k, c)."""
    k = A.shape[0]
    out = np.zeros((A.shape[1], V.shape[1]), dtype=np.longdouble)
    err = np.zeros(out.shape)
    for k0 in range(0, k, KB):
        a, v = A[k0:k0 + KB], V[k0:k0 + KB]
        out += a.T.astype(np.longdouble) @ v.astype(np.longdouble)
        err += 192 * 2.0 ** -55 * np.abs(a).max(0)[:, None] * np.abs(v).astype(float).max(0)[None, :]
    return out, err + (k / KB + 3) * 2.0 ** -53 * (np.abs(A).T @ np.abs(V).astype(float))


def reference(Uout, S, Uin, V):
    W, e1 = contract(Uin, V)
    W = S[:, None] * W
    Y, e2 = contract(np.ascontiguousarray(Uout.T), W)
    e1 = np.abs(S)[:, None] * e1 + 2.0 ** -52 * np.abs(W).astype(float)
    return Y, e2 + np.abs(Uout) @ e1


@pytest.mark.parametrize("d,n,tol", [(3, 256, 1e-6), (3, 257, 1e-4), (4, 383, 1e-3), (3, 1000, 1e-7),
                                     (5, 2049, 1e-2)])
def test_products_match_extended_precision(d, n, tol):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(10 * n + d)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), "gaussian", 0.8, tol)
    assert f.info.ldu >= 64
    U, S = f.export()
    for c in (5, 16, 17, 33):
        V = g.standard_normal((n, c)) * np.exp(g.uniform(-20, 20, (n, 1)))
        V[:, 0] = 0.0                                  # a zero column
        V[:, 1] = 0.0
        V[n // 2, 1] = 1.0                             # a unit vector
        V[:, 2] = 0.9999                               # every digit sum of one sign
        V[: n // 2, 3] = 0.0                           # whole blocks of zeros
        V[:, 4] *= 1e-200
        Y = f.matvec(to_dev(V)).cpu().numpy()
        ref, bound = reference(U, S, U, V)
        assert np.all(Y[:, 0] == 0.0)
        assert np.all(np.abs(Y - ref) <= bound), c
    # a group of 64, then one of 5
    V = g.standard_normal((n, 69))
    Y = f.matvec(to_dev(V)).cpu().numpy()
    ref, bound = reference(U, S, U, V)
    assert np.all(np.abs(Y - ref) <= bound)


def test_cross_and_solve_and_nan():
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(3)
    x, y = g.uniform(-1, 1, (1201, 3)), g.uniform(-1, 1, (640, 3))
    f = hdf.build_cross(to_dev(x), to_dev(y), "cauchy", 1.0, 1e-6)
    U, S = f.export()
    V = f.export_y()
    B, W = g.standard_normal((640, 9)), g.standard_normal((1201, 9))
    for out, (ref, bound) in ((f.matvec(to_dev(B)), reference(U, S, V, B)),
                              (f.matvec_t(to_dev(W)), reference(V, S, U, W))):
        assert np.all(np.abs(out.cpu().numpy() - ref) <= bound)
    B[100, 3] = np.nan
    B[5, 4] = np.inf
    out = f.matvec(to_dev(B)).cpu().numpy()
    assert np.isnan(out[:, 3]).all() and np.isnan(out[:, 4]).all()
    assert np.isfinite(np.delete(out, [3, 4], axis=1)).all()
    # many right-hand sides of a solve give what single ones (the streaming kernels) give
    h = hdf.build(to_dev(x), "gaussian", 0.7, 1e-6)
    X = h.solve(0.1, to_dev(W), refine_steps=1).cpu().numpy()
    for j in (0, 8):
        x1 = h.solve(0.1, to_dev(W[:, j]), refine_steps=1).cpu().numpy()
        assert np.linalg.norm(X[:, j] - x1) <= 1e-9 * np.linalg.norm(x1)


def test_cuda_core_flag_and_agreement_at_size():
    """20,001 points, rank about 10^4: tensor cores against the CUDA-core form of the same factor."""
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as Wl
    x = to_dev(Wl.points("mixture3_matern", n=20001))
    f = hdf.build(x, "matern32", 1.0, 1e-8)
    h = hdf.build(x, "matern32", 1.0, 1e-8, flags=hdf.FLAG_CUDA_CORES)
    V = torch.randn(20001, 40, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    a, b = f.matvec(V), h.matvec(V)
    assert float((a - b).norm() / b.norm()) <= 1e-13
