"""The stored off-diagonal blocks of the regression operator at the edges of their tiles, and the
conjugate gradients that run on the device.

Bound: FP32 coordinates shifted by a data point (differences below 2, relative error 2^-23 each)
and an FP32 kernel value err by at most 8 2^-22 per entry for d <= 8 and l = 0.5 (the exponent
0.5 z^2 <= 16 is off by 16 2^-22 / 8 where the value is not small); the diagonal blocks by tol times
their Frobenius norm."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


def dense(x, ell):
    d2 = ((x[:, None, :] - x[None, :, :]) ** 2).sum(-1)
    return np.exp(-0.5 * d2 / ell ** 2)


@pytest.mark.parametrize("n,d,clusters", [(5, 3, 2), (127, 4, 3), (129, 8, 1), (1023, 5, 4), (1025, 5, 7), (1026, 3, 5)])
def test_operator_and_solve_against_dense(n, d, clusters):
    import torch
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(n)
    x = g.uniform(0, 1, (n, d))
    lab = g.integers(0, clusters, n)
    tol = 1e-6
    m = hdf.KRR(to_dev(x), torch.from_numpy(lab).cuda(), "gaussian", 0.5, 1.0, tol)
    K = dense(x, 0.5)
    v = g.standard_normal(n)
    y = m.apply(to_dev(v)).cpu().numpy()
    bound = 32 * 2.0 ** -22 * np.abs(v).sum() + tol * n * np.linalg.norm(v)
    assert np.abs(y - (v + K @ v)).max() <= bound
    # the operator is one fixed symmetric matrix
    w = g.standard_normal(n)
    z = m.apply(to_dev(w)).cpu().numpy()
    assert abs(w @ y - v @ z) <= 1e-12 * np.linalg.norm(w) * np.linalg.norm(y) * np.sqrt(n)
    # conjugate gradients reach their tolerance on it, and stop at the same state when asked again
    a, it, res = m.solve(to_dev(v), rtol=1e-10, max_iter=2000)
    r = v - m.apply(a).cpu().numpy()
    assert res <= 1e-10 and np.linalg.norm(r) <= 1e-8 * np.linalg.norm(v)
    b, it2, res2 = m.solve(to_dev(v), rtol=1e-10, max_iter=2000)
    assert it2 == it and res2 == res and bool((a == b).all())
    # too few iterations: the count is the limit and the status says so
    if it > 2:
        c, itc, resc = m.solve(to_dev(v), rtol=1e-10, max_iter=2)
        assert itc == 2 and resc > 1e-10 and m.status in (0, 4)
    z0, it0, res0 = m.solve(torch.zeros(n, dtype=torch.float64, device="cuda"))
    assert it0 == 0 and res0 == 0.0 and bool((z0 == 0).all())
