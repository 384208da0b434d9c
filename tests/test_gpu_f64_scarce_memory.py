"""FP64 products whose work space cannot be had go on in a form that needs less: tensor-core slices, then
the streaming kernels, then the register-tiled ones.  Only W itself cannot be done without.  Each form is
within k 2^-53 of the sums of magnitudes for a contraction of length k."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu
ENOMEM = 2


@pytest.mark.parametrize("d,n,tol", [(3, 300, 1e-5), (4, 2049, 1e-4)])
def test_products_without_work_space(d, n, tol):
    import torch
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(n)
    f = hdf.build(to_dev(g.uniform(-1, 1, (n, d))), "gaussian", 0.8, tol)
    assert f.info.ldu >= 64
    U, S = (torch.from_numpy(a).cuda() for a in f.export())
    for c in (1, 3, 5, 17, 40, 69):
        V = torch.from_numpy(g.standard_normal((c, n))).cuda()
        ref = (U @ (S[:, None] * (U.T @ V.T))).T
        mag = (U.abs() @ (S.abs()[:, None] * (U.abs().T @ V.abs().T))).T
        failed = 0
        try:
            for k in range(16):
                Y = torch.full_like(V, 3.0)
                hdf.debug_fail_alloc(k)
                try:
                    f.matvec_ptr(V.data_ptr(), n, c, Y.data_ptr(), n)
                except hdf.HdfError as e:
                    assert e.status == ENOMEM and bool((Y == 3.0).all())
                    failed += 1
                    continue
                finally:
                    hdf.debug_fail_alloc(-1)
                assert bool(((Y - ref).abs() <= 2 * (n + f.rank) * 2.0 ** -53 * mag).all()), (c, k)
                assert f.device_errors() == 0
        finally:
            hdf.debug_fail_alloc(-1)
        assert failed == 1, (c, failed)
