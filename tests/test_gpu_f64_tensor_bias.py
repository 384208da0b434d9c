"""The block sums of the FP64 slice products carry no error of one sign.

With blocks of 64 along the contraction the sum of a block is an integer in units of 2^(eu + ev - 54), eu
and ev the exponents of the block's largest values (|x| < 2^e).  Cut off towards minus infinity it would
be short by half a unit on average whatever its sign, and W = U^T V by the sum of those over the blocks.
Here the points come in equal pairs with V = (v, -v (1 + 2^-30 t)), so that the sums themselves are small
and their own FP64 rounding does not hide the effect.  The error of Y = U S W is projected on what that
shortfall would give: 1 for cutting off, 0 for rounding.  Spread: rounding (half a unit uniformly,
0.58 of the shortfall) and the truncated operands (at most as much again for 32 pairs) are independent
from block to block; over 256 blocks at most 1.2 / 16 = 0.08 if all columns went together."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


def exponent(a):
    """e with |a| < 2^e and 2^(e - 1) <= |a|."""
    return np.frexp(a)[1]


@pytest.mark.parametrize("d,tol,c", [(3, 1e-4, 5), (3, 1e-4, 17), (4, 1e-3, 8)])
def test_mean_error_over_blocks(d, tol, c):
    from paper_2202_03655_gb300 import hdf
    n = 16384
    g = np.random.default_rng(d + c)
    x = np.repeat(g.uniform(-1, 1, (n // 2, d)), 2, axis=0)
    f = hdf.build(to_dev(x), "gaussian", 0.8, tol)
    U, S = f.export()
    assert f.info.ldu >= 64 and bool((U[0::2] == U[1::2]).all())
    v = g.standard_normal((n // 2, c))
    V = np.empty((n, c))
    V[0::2], V[1::2] = v, -v * (1.0 + 2.0 ** -30 * g.uniform(0.5, 1.5, v.shape))
    Y = f.matvec(to_dev(V)).cpu().numpy()
    UL, VL = U.astype(np.longdouble), V.astype(np.longdouble)
    err = (Y - UL @ (S[:, None] * (UL.T @ VL))).astype(np.float64)
    eu = exponent(np.abs(U).reshape(n // 64, 64, -1).max(1))
    ev = exponent(np.abs(V).reshape(n // 64, 64, -1).max(1))
    short = -(2.0 ** (eu[:, :, None] + ev[:, None, :] - 55.0)).sum(0)
    b = U @ (S[:, None] * short)
    coef = (err * b).sum() / (b * b).sum()
    print("projection", coef)
    assert abs(coef) <= 0.25
