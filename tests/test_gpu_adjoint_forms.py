"""The adjoint's table layouts, batches and CTA sizes: high degrees (few warps per SM: three arrays, CTAs
of one or two warps) and low ones (packed, four warps), at numbers of points that take batches of one,
two and four.

Batches: `copies` equal copies of m points have the centre, radius and kernel means of the m points, and
their factor restricted to one copy is that of the m points, so with v and w on one copy of each point the
gradient there is the m points' own, and zero elsewhere.  The two builds differ by the rounding of
their bases; a derivative of a degree-L polynomial magnifies that by at most L^2: L^2 times some tens of
units of the bulk precision."""
import numpy as np
import pytest

from gpu_common import rel, to_dev
from oracle import hdf as ohdf

pytestmark = pytest.mark.gpu

CASES = [(3, "gaussian", 0.22, 1e-8), (4, "gaussian", 0.3, 1e-6), (3, "gaussian", 0.8, 1e-6), (5, "cauchy", 1.5, 1e-4),
         (7, "gaussian", 1.5, 1e-4), (8, "gaussian", 2.0, 1e-4)]


def points(m, d):
    g = np.random.default_rng(10 * m + d)
    x = g.standard_normal((m, d))
    x *= (g.random(m) ** (1.0 / d) / np.linalg.norm(x, axis=1))[:, None]
    return g, x


@pytest.mark.parametrize("d,kname,ell,tol", CASES)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_against_the_exact_kernel(d, kname, ell, tol, prec):
    import torch
    from paper_2202_03655_gb300 import hdf
    g, x = points(1500, d)
    v, w = g.standard_normal(1500), g.standard_normal(1500)
    dt = torch.float64 if prec == "fp64" else torch.float32
    f = hdf.build(to_dev(x), kname, ell, tol, precision=prec)
    G, _, _ = f.adjoint(to_dev(x), to_dev(v, dt), to_dev(w, dt))
    Go = ohdf.dense_gradient(x, kname, ell, v, w)[0]
    L = f.info.p // 2
    # the approximation's error and the bulk rounding, both magnified by the derivative
    assert rel(G.double().cpu().numpy(), Go) <= L * L * (10 * tol + (32 * 2.0 ** -24 if prec == "fp32" else 0.0))


@pytest.mark.parametrize("d,kname,ell,tol", CASES)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("copies", [41, 83])
def test_copies_of_points(d, kname, ell, tol, prec, copies):
    import torch
    from paper_2202_03655_gb300 import hdf
    m = 500
    g, x = points(m, d)
    dt = torch.float64 if prec == "fp64" else torch.float32
    v, w = to_dev(g.standard_normal(m), dt), to_dev(g.standard_normal(m), dt)
    f = hdf.build(to_dev(x), kname, ell, tol, precision=prec)
    G, _, _ = f.adjoint(to_dev(x), v, w)
    h = hdf.build(to_dev(np.repeat(x, copies, axis=0)), kname, ell, tol, precision=prec)
    assert h.info.p == f.info.p
    at = torch.from_numpy(np.arange(m) * copies + g.integers(0, copies, m)).cuda()
    V, W = (torch.zeros(m * copies, dtype=dt, device="cuda").index_put_((at,), a) for a in (v, w))
    H, _, _ = h.adjoint(to_dev(np.repeat(x, copies, axis=0)), V, W)
    eps = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    L = f.info.p // 2
    assert rel(H[at].double().cpu().numpy(), G.double().cpu().numpy()) <= 64 * L * L * eps + tol
    H[at] = 0
    assert bool((H == 0).all())
