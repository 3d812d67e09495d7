"""Kernel k-means++ on rows that repeat: the distance of a row that equals a
chosen one is exactly 0, whatever the kernel, so a chosen row is not drawn again
while others are left, and draws are uniform once every distinct row is chosen."""
import numpy as np
import pytest

from oracle.init import uniform01
from oracle.rng import index_below, splitmix64

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["linear", "poly", "gaussian", "laplacian"])
@pytest.mark.parametrize("d", [65, 784])
@pytest.mark.parametrize("n", [300, 50_000])
def test_two_distinct_rows(kernel, d, n):
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import kmeanspp
    rng = np.random.default_rng(d + n)
    rows = rng.normal(size=(2, d)).astype(np.float32)
    which = rng.integers(0, 2, size=n)
    for seed in (1, 2, 3):
        got = kmeanspp(torch.from_numpy(rows[which]).cuda(), 6, kernel, 2.0 * d, coef0=1.0, degree=2, seed=seed)
        assert got[0] == index_below(splitmix64(seed, 0), n)
        # draw 1: every other row has the same D^2, so the target's rank among them is floor(u count)
        others = np.flatnonzero(which != which[got[0]])
        rank = uniform01(seed, 1) * len(others)
        assert abs(rank - round(rank)) > 1e-6
        assert got[1] == others[int(rank)]
        for t in range(2, 6):                  # every distance is 0
            assert got[t] == index_below(splitmix64(seed, t), n)
