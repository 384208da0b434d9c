"""Batches in which some sets keep no column.  A nearly constant kernel (lengthscale 30) has the trace n
and mean square 1, so a truncation budget 0.5 eta tol n sqrt(mu2) above n drops all of it; at
lengthscale 0.3 the budget is far below the trace.  The sets with columns give what each gives on its own:
the two forms add the same products in different orders, the bound is that of the rounding."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu

SIZES = [37, 150, 37, 257, 64, 400, 5]
ELLS = [30.0, 0.3, 30.0, 0.3, 30.0, 0.3, 30.0]


def batch(prec):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(2)
    off = np.concatenate([[0], np.cumsum(SIZES)])
    x = g.uniform(-0.5, 0.5, (off[-1], 3))
    b = hdf.build_batched(to_dev(x), off, "gaussian", ELLS, 0.6, precision=prec, eta=4.0)
    assert [b.info(s).rank == 0 for s in range(len(SIZES))] == [e == 30.0 for e in ELLS]
    return b, x, off


@pytest.mark.parametrize("prec,eps", [("fp64", 2.0 ** -53), ("fp32", 2.0 ** -24)])
def test_sets_with_columns(prec, eps):
    import torch
    b, x, off = batch(prec)
    dt = torch.float64 if prec == "fp64" else torch.float32
    for c in (1, 2, 3, 4, 5, 8, 12, 17):
        V = torch.randn(int(off[-1]), c, dtype=dt, device="cuda", generator=torch.Generator("cuda").manual_seed(c))
        Y = b.matvec(V)
        for s, (lo, hi) in enumerate(zip(off[:-1], off[1:])):
            if ELLS[s] == 30.0:
                continue
            U, S = (torch.from_numpy(np.asarray(a, dtype=np.float64)).cuda() for a in b.export(s))
            v = V[lo:hi].double()
            ref = U @ (S[:, None] * (U.T @ v))
            bound = 4 * (hi - lo) * eps * (U.abs() @ (S.abs()[:, None] * (U.abs().T @ v.abs())))
            assert bool(((Y[lo:hi].double() - ref).abs() <= bound).all()), (c, s)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_sets_without_columns_give_zero(prec):
    import torch
    b, x, off = batch(prec)
    n, dt = int(off[-1]), torch.float64 if prec == "fp64" else torch.float32
    for c in (1, 3, 8, 17):
        V = torch.ones(c, n, dtype=dt, device="cuda")
        Y = torch.full((c, n + 3), 7.0, dtype=dt, device="cuda")       # longer columns than the points
        b.matvec_ptr(V.data_ptr(), n, c, Y.data_ptr(), n + 3)
        for s, (lo, hi) in enumerate(zip(off[:-1], off[1:])):
            assert bool((Y[:, lo:hi] == 0.0).all()) == (ELLS[s] == 30.0), (c, s)
        assert bool((Y[:, n:] == 7.0).all())
