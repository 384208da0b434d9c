"""Rows whose harmonics do not fit a warp's share of shared memory (formed as products per column),
against the dense kernel, single and batched.

Bound: |K~ - K|_F <= tol |K|_F (a build that reached its tolerance), plus the rounding of the rows:
an entry of U is a product of at most d - 1 level values, each off by a few roundings of
recurrences of length <= L, times a radial factor, together 256 eps, so |U S U^T V| moves by at
most 2 x 256 eps |U| |S| |U|^T |V| (both sides), and the product adds less than that."""
import numpy as np
import pytest

from gpu_common import to_dev
from oracle.kernels import kernel

pytestmark = pytest.mark.gpu


def dense(x, ell):
    return kernel("gaussian", np.linalg.norm(x[:, None, :] - x[None, :, :], axis=-1), ell)


def check(f, x, ell, tol, eps, V, Y):
    K = dense(x, ell)
    U, S = f.export()
    A = np.abs(U.astype(np.float64))
    rows = 1024 * eps * (A @ (np.abs(S.astype(np.float64))[:, None] * (A.T @ np.abs(V))))
    assert np.linalg.norm(Y - K @ V) <= tol * np.linalg.norm(K) * np.linalg.norm(V) + np.linalg.norm(rows)


# ranks 3,584 (slots) and, as products: descriptors per column, per chunk, in global memory
@pytest.mark.parametrize("d,ell,tol,precision", [
    (4, 0.3, 1e-5, "fp32"), (4, 0.3, 1e-10, "fp32"), (5, 0.5, 1e-8, "fp32"), (5, 0.3, 1e-5, "fp32"),
    (5, 0.3, 1e-8, "fp32"), (5, 0.3, 1e-10, "fp32"),
    (4, 0.3, 1e-8, "fp64"), (5, 0.5, 1e-8, "fp64"), (5, 0.5, 1e-10, "fp64"), (5, 0.3, 1e-6, "fp64")])
@pytest.mark.parametrize("n", [3, 157])
def test_row_products(d, ell, tol, precision, n):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(10 * d + n)
    x = g.random((n, d))
    if n > 3:
        x[5] = x[6]
        x[9, 2:] = 0.5
    f = hdf.build(to_dev(x), "gaussian", ell, tol, precision=precision)
    V = g.standard_normal((n, 2))
    vt = to_dev(V) if precision == "fp64" else to_dev(V).float()
    check(f, x, ell, tol, 2.0 ** (-53 if precision == "fp64" else -24), V, f.matvec(vt).double().cpu().numpy())


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_batched_row_products(precision):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(3)
    sizes, ells, tol = [90, 33, 140], [2.0, 0.5, 0.4], 1e-6
    x = np.concatenate([g.random((n, 5)) for n in sizes])
    off = np.concatenate([[0], np.cumsum(sizes)])
    b = hdf.build_batched(to_dev(x), off, "gaussian", ells, tol, precision=precision)
    V = g.standard_normal((len(x), 2))
    vt = to_dev(V) if precision == "fp64" else to_dev(V).float()
    Y = b.matvec(vt).double().cpu().numpy()
    for s, ell in enumerate(ells):
        q = slice(off[s], off[s + 1])
        K = dense(x[q], ell)
        # entries of K~ are below 2 and the rows of U S U^T hold them as sums of like magnitude
        slack = (0.0 if precision == "fp64" else 1024 * 2.0 ** -24 * sizes[s])
        assert np.linalg.norm(Y[q] - K @ V[q]) <= (tol * np.linalg.norm(K) + slack) * np.linalg.norm(V[q])


# degrees below 8, 8 to 15 and above (groups of 8, 16 and 32 lanes per point), with points that leave
# groups of the last warp without one
@pytest.mark.parametrize("d,ell,tol,lo,hi", [(3, 2.0, 1e-6, 1, 8), (3, 0.6, 1e-6, 8, 16), (3, 0.2, 1e-6, 16, 33),
                                             (4, 1.0, 1e-4, 1, 8), (4, 0.5, 1e-5, 8, 16), (5, 0.6, 1e-3, 1, 16),
                                             (8, 2.0, 1e-2, 1, 8)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [1, 2, 5, 67])
def test_lane_groups(d, ell, tol, lo, hi, precision, n):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(10 * d + n)
    x = g.random((n, d))
    x *= np.sqrt(3.0 / d)
    if n > 3:
        x[2, 2:] = x[3, 2:]
    f = hdf.build(to_dev(x), "gaussian", ell, tol, precision=precision)
    if n == 67:
        assert lo <= max(k for k, s in enumerate(f.s_k) if s) < hi
    V = g.standard_normal((n, 2))
    vt = to_dev(V) if precision == "fp64" else to_dev(V).float()
    check(f, x, ell, tol, 2.0 ** (-53 if precision == "fp64" else -24), V, f.matvec(vt).double().cpu().numpy())
    b = hdf.build_batched(to_dev(np.concatenate([x, x])), [0, n, 2 * n], "gaussian", [ell, ell], tol, precision=precision)
    Y = b.matvec(to_dev(np.concatenate([V, V])).to(vt.dtype)).double().cpu().numpy()
    check(f, x, ell, tol, 2.0 ** (-53 if precision == "fp64" else -24), V, Y[:n])
    assert np.array_equal(Y[:n], Y[n:])
