"""The reductions of the partial sums of U^T V at the sizes where their forms change: few and many row
chunks, few and many results, narrow and wide blocks of columns, ranks that end inside a tile.

Bound: K~V against the exported factor in FP64: both contractions round (k + 64) units of the bulk
precision of the sums of magnitudes (the slices themselves are summed in FP64)."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,kname,tol", [(4, 300, "matern32", 1e-3), (3, 900, "gaussian", 1e-7),
                                          (4, 6001, "gaussian", 1e-4), (5, 700, "matern32", 1e-2)])
@pytest.mark.parametrize("prec,flags", [("fp64", 0), ("fp32", 0), ("fp64", 1), ("fp32", 1)])
def test_products_against_the_factor(d, n, kname, tol, prec, flags):
    import torch
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(n)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), kname, 0.8, tol, precision=prec, flags=flags)
    U, S = (torch.from_numpy(np.asarray(a, dtype=np.float64)).cuda() for a in f.export())
    eps, dt = (2.0 ** -53, torch.float64) if prec == "fp64" else (2.0 ** -24, torch.float32)
    for c in (1, 3, 5, 16, 33, 47, 48, 49, 64, 65):
        V = to_dev(g.standard_normal((n, c)), dt)
        v = V.double()
        ref = U @ (S[:, None] * (U.T @ v))
        mag = U.abs() @ (S.abs()[:, None] * (U.abs().T @ v.abs()))
        err = (f.matvec(V).double() - ref).abs()
        assert bool((err <= (n + f.rank + 64) * eps * mag).all()), c
