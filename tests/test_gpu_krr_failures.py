"""Builds of the regression operator that fail on the host: a singular block and device allocations
that report out-of-memory.  Each returns its status, hands back no model and leaves the library usable:
the next build, product and solve give what they give without a failure before them."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu
ENOMEM, ESINGULAR = 2, 6


def problem(n=900, clusters=4):
    import torch
    g = np.random.default_rng(5)
    x = g.uniform(0, 1, (n, 4))
    return x, torch.from_numpy(g.integers(0, clusters, n)).cuda(), to_dev(g.standard_normal(n))


def build(x, lab, lam=1.0):
    from paper_2202_03655_gb300 import hdf
    return hdf.KRR(to_dev(x), lab, "gaussian", 0.5, lam, 1e-6)


def test_singular_block():
    from paper_2202_03655_gb300 import hdf
    x, lab, v = problem()
    m = build(x, lab)
    y, w = m.apply(v), m.solve(v, rtol=1e-8)[0]
    xs = x.copy()
    first = np.flatnonzero(lab.cpu().numpy() == lab.cpu().numpy()[0])
    xs[first[1]] = xs[first[0]]              # two equal points of one cluster: rows of K_cc repeat
    for _ in range(3):
        with pytest.raises(hdf.HdfError) as ei:
            build(xs, lab, 1e-20)            # 1 + 1e-20 = 1: the second pivot is zero
        assert ei.value.status == ESINGULAR
    m2 = build(x, lab)
    assert bool((m2.apply(v) == y).all())
    assert bool((m2.solve(v, rtol=1e-8)[0] == w).all())


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_injected_allocation_failures(prec):
    from paper_2202_03655_gb300 import hdf
    x, lab, v = problem()
    xt = to_dev(x)
    ref = hdf.KRR(xt, lab, "gaussian", 0.5, 1.0, 1e-6, precision=prec)
    y, w = ref.apply(v), ref.solve(v, rtol=1e-8)[0]
    failed = 0
    try:
        for k in range(80):                  # a build makes some forty allocations
            hdf.debug_fail_alloc(k)
            try:
                m = hdf.KRR(xt, lab, "gaussian", 0.5, 1.0, 1e-6, precision=prec)
            except hdf.HdfError as e:
                assert e.status == ENOMEM, (k, str(e))
                failed += 1
                continue
            hdf.debug_fail_alloc(-1)
            # built all the same: past the last allocation, or without the stored blocks, whose
            # evaluated form adds the same FP32 values in another order
            assert float((m.apply(v) - y).abs().max()) <= 1e-9 * float(v.abs().sum())
            m.free()
    finally:
        hdf.debug_fail_alloc(-1)
    assert failed >= 20
    m = hdf.KRR(xt, lab, "gaussian", 0.5, 1.0, 1e-6, precision=prec)
    assert bool((m.apply(v) == y).all())
    assert bool((m.solve(v, rtol=1e-8)[0] == w).all())


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_stored_blocks_are_given_up_for_any_allocation_of_theirs(prec):
    """A build without memory for the stored blocks or for their partial sums evaluates the blocks instead."""
    from paper_2202_03655_gb300 import hdf
    x, lab, v = problem()
    xt = to_dev(x)
    y = hdf.KRR(xt, lab, "gaussian", 0.5, 1.0, 1e-6, precision=prec).apply(v)
    other = 0
    try:
        for k in range(80):
            hdf.debug_fail_alloc(k)
            try:
                m = hdf.KRR(xt, lab, "gaussian", 0.5, 1.0, 1e-6, precision=prec)
            except hdf.HdfError:
                continue
            hdf.debug_fail_alloc(-1)
            z = m.apply(v)
            w, it, res = m.solve(v, rtol=1e-8)
            assert res <= 1e-8
            # evaluated: the same FP32 values added in another order
            other += not bool((z == y).all())
            assert float((z - y).abs().max()) <= 1e-9 * float(v.abs().sum())
    finally:
        hdf.debug_fail_alloc(-1)
    assert other == 2
