"""FP64 products of few columns (streaming kernels) against numpy on the exported factor, at the
edges of their row groups, column steps, row chunks and column counts.

Bound: every entry of U (S (U^T V)) is a sum of n r products of three rounded factors, so in any
order of summation |error| <= 2 (n + r + 4) eps |U| |S| |U|^T |V| entrywise."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,tol", [(3, 1, 1e-6), (3, 7, 1e-6), (3, 9, 1e-8), (4, 255, 1e-3), (3, 2001, 1e-6),
                                     (5, 513, 1e-5), (4, 4099, 1e-4)])
def test_few_columns_match_numpy(d, n, tol):
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(100 * d + n)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), "gaussian", 0.7, tol)
    U, S = f.export()
    aU = np.abs(U)
    for c in (1, 2, 3, 4, 5, 65, 67):          # 65 and 67: a group of 64, then one or three columns
        V = g.standard_normal((n, c)) * np.exp(g.uniform(-5, 5, (n, 1)))
        Y = f.matvec(to_dev(V)).cpu().numpy()
        ref = U @ (S[:, None] * (U.T @ V))
        bound = 2 * (n + f.rank + 4) * 2.0 ** -53 * (aU @ (np.abs(S)[:, None] * (aU.T @ np.abs(V))))
        assert np.all(np.abs(Y - ref) <= 2 * bound), c      # twice: numpy's own error


def test_few_columns_cross_and_infinities():
    """Both directions of a cross factor, and a non-finite entry reaches every row it should."""
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(5)
    x, y = g.uniform(-1, 1, (1201, 3)), g.uniform(-1, 1, (333, 3))
    f = hdf.build_cross(to_dev(x), to_dev(y), "cauchy", 1.0, 1e-6)
    U, S = f.export()
    V = f.export_y()
    for c in (1, 3):
        B, W = g.standard_normal((333, c)), g.standard_normal((1201, c))
        for out, ref in ((f.matvec(to_dev(B)), U @ (S[:, None] * (V.T @ B))),
                         (f.matvec_t(to_dev(W)), V @ (S[:, None] * (U.T @ W)))):
            out = out.cpu().numpy()
            assert np.linalg.norm(out - ref) <= 1e-12 * np.linalg.norm(ref)
    b = np.ones(333)
    b[17] = np.nan
    assert np.isnan(f.matvec(to_dev(b)).cpu().numpy()).all()


@pytest.mark.parametrize("c", [1, 2, 3, 4, 5])
def test_batched_sets_match_single_builds(c):
    """FP64 batches of few columns: ragged sets (below, at and above one chunk and one row block)
    against the same sets built alone, whose products are checked above."""
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(77)
    sizes = [1, 7, 63, 64, 65, 300, 2049, 5000]
    off = np.concatenate([[0], np.cumsum(sizes)])
    x = g.uniform(-1, 1, (off[-1], 3))
    ells = g.uniform(0.5, 1.0, len(sizes))
    V = g.standard_normal((off[-1], c))
    Y = hdf.build_batched(to_dev(x), off, "gaussian", ells, 1e-6, precision="fp64").matvec(to_dev(V)).cpu().numpy()
    for s in range(len(sizes)):
        sl = slice(off[s], off[s + 1])
        y = hdf.build(to_dev(x[sl]), "gaussian", ells[s], 1e-6).matvec(to_dev(V[sl])).cpu().numpy()
        assert np.linalg.norm(Y[sl] - y) <= 10e-6 * np.linalg.norm(y)      # two factors of the same tolerance
