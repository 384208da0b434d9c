"""k-means where a block takes several chunks of points, and the work space it may take.

Bounds: a centre is a sum of at most n coordinates below 1 in magnitude divided by their number; sums of
two orders differ by at most 2 n 2^-53 of the sum of magnitudes, so centres by 2 n 2^-53."""
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("n,d,k", [(65535, 3, 5), (65537, 8, 9), (131073, 1, 300), (200001, 5, 1), (196608, 8, 768)])
def test_one_pass_against_sums(n, d, k):
    import torch
    from paper_2202_03655_gb300 import hdf
    g = np.random.default_rng(n)
    x = to_dev(g.uniform(-1, 1, (n, d)))
    init = np.sort(g.choice(n, k, replace=False))
    labels, C, it = hdf.kmeans(x, init, max_iter=1)
    lab = labels.long()
    # nearest centre: no other is closer by more than the rounding of a distance
    d2 = ((x[:, None, :] - x[torch.from_numpy(init).cuda()][None]) ** 2).sum(-1)
    own = d2.gather(1, lab[:, None])[:, 0]
    assert it == 1 and bool((own <= d2.amin(1) * (1 + 32 * 2.0 ** -52)).all())
    cnt = torch.bincount(lab, minlength=k).double()
    ref = torch.stack([torch.bincount(lab, weights=x[:, j], minlength=k) for j in range(d)], 1) / cnt[:, None]
    assert bool((cnt > 0).all()) and float((C - ref).abs().max()) <= 2 * n * 2.0 ** -53
    again = hdf.kmeans(x, init, max_iter=1)
    assert bool((again[0] == labels).all()) and bool((again[1] == C).all())


def test_work_space_does_not_grow_with_the_points():
    """1,000,000 points in 600 clusters, d = 8: 512 blocks' sums are 22 MB (a block per 128 points 337 MB)."""
    code = """
import torch
from paper_2202_03655_gb300 import hdf
x = torch.rand(1_000_000, 8, dtype=torch.float64, device="cuda")
hdf.kmeans(x[:5000].contiguous(), range(600), max_iter=1)
labels = torch.empty(1_000_000, dtype=torch.int32, device="cuda")
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
hdf.kmeans(x, range(600), max_iter=1)
torch.cuda.synchronize()
print("grew", free - torch.cuda.mem_get_info()[0])
"""
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    grew = int(out.stdout.split("grew")[1])
    # the sums, the labels that the binding returns and the pools' granularity (torch 20 MiB, CUDA 32 MiB)
    assert grew <= 512 * 600 * 9 * 8 + (4 + 20 + 2 * 32) * 2 ** 20, grew
