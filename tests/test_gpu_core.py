"""The core of the Woodbury solve: the factorization without pivoting at the edges of its 64-wide
tiles, and the pivoted LU that takes over when lambda I + K~ is indefinite.

Both are backward stable on the core, so the solution X of (lambda I + K~) X = B leaves a residual of
a modest multiple of r eps |A| |X|; the factor 64 covers the growth of the products U C^-1 U^T
(|U| <= 1) divided by lambda."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


def check(f, lam, c, seed, refine):
    U, S = f.export()
    n = U.shape[0]
    B = np.random.default_rng(seed).standard_normal((n, c))
    X = f.solve(lam, to_dev(B), refine_steps=refine).cpu().numpy()
    A = (U * S) @ U.T + lam * np.eye(n)
    R = A @ X - B
    an = np.linalg.norm(A, 2)
    assert np.linalg.norm(R) <= 64 * f.info.ldu * 2.0 ** -53 * an / lam * np.linalg.norm(B)
    return np.linalg.eigvalsh(A)[0]


@pytest.mark.parametrize("d,n,tol", [(3, 40, 1e-2), (3, 300, 1e-3), (3, 700, 1e-5), (3, 901, 1e-6), (4, 600, 1e-4)])
@pytest.mark.parametrize("c", [1, 3, 64, 65])
def test_definite_systems(d, n, tol, c):
    from paper_2202_03655_gb300 import hdf
    x = np.random.default_rng(n).uniform(-1, 1, (n, d))
    f = hdf.build(to_dev(x), "gaussian", 0.7, tol)
    assert check(f, 0.5, c, 1, 1) > 0


@pytest.mark.parametrize("n,p_max", [(400, 8), (900, 10)])
def test_indefinite_systems_fall_back(n, p_max):
    """At a capped degree with fewer columns than points K~ has as many negative eigenvalues as S
    has negative entries (Sylvester); a lambda below them makes the system indefinite, which the
    pivoted LU solves.  Then a definite lambda on the same factor."""
    from paper_2202_03655_gb300 import hdf
    x = np.random.default_rng(n).uniform(-1, 1, (n, 3))
    f = hdf.build(to_dev(x), "matern32", 0.5, 1e-6, p_max=p_max)
    U, S = f.export()
    assert f.rank < n and S.min() < 0
    ev = np.linalg.eigvalsh((U * S) @ U.T)
    assert ev[0] < -1e-6
    lam = 0.5 * abs(ev[0])
    n_B = np.random.default_rng(2).standard_normal((n, 2))
    X = f.solve(lam, to_dev(n_B), refine_steps=1).cpu().numpy()
    A = (U * S) @ U.T + lam * np.eye(n)
    smin = np.abs(np.linalg.eigvalsh(A)).min()
    assert np.linalg.norm(A @ X - n_B) <= 64 * f.info.ldu * 2.0 ** -53 * np.linalg.norm(A, 2) / min(lam, smin) * \
        np.linalg.norm(n_B)
    assert check(f, 4.0 * abs(ev[0]), 2, 3, 1) > 0


def test_gram_is_symmetric_and_right():
    """The mirrored Gram through an FP32 solve with many right-hand sides, at a width that is no
    multiple of the 64-column blocks."""
    from paper_2202_03655_gb300 import hdf
    import torch
    g = np.random.default_rng(8)
    x = to_dev(g.uniform(-1, 1, (3001, 4)))
    f = hdf.build(x, "gaussian", 0.8, 1e-4, precision="fp32")
    h = hdf.build(x, "gaussian", 0.8, 1e-4, precision="fp64")
    assert f.info.ldu % 64 != 0
    B = to_dev(g.standard_normal((3001, 5)))
    X = f.solve(10.0, B.float(), refine_steps=1).double()
    Y = h.solve(10.0, B, refine_steps=1)
    assert float((X - Y).norm() / Y.norm()) <= 1e-4       # FP32 factor: eps32 |A| / lambda
