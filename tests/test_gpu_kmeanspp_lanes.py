"""Kernel k-means++ with one, two, four and eight lanes a point: few points with
many features, remainders of the points per block and of the lanes' feature
tiles, aligned and unaligned rows. The chosen indices must equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2410_05902_gb300 import inputs

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["gaussian", "laplacian", "linear", "poly"])
@pytest.mark.parametrize("n,d,pad", [
    (5001, 33, 0),      # two lanes
    (5001, 68, 4),      # four lanes, 16-byte loads
    (4999, 129, 0),     # eight lanes
    (17, 784, 0),
    (3, 300, 1),
    (20_001, 300, 0),   # two lanes: the points fill the rest
    (9999, 300, 0),     # four
    (40_001, 70, 0),    # one
    (60, 4096, 0),      # the widest rows
])
def test_lanes_match_oracle(kernel, n, d, pad):
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import kmeanspp
    X, _ = inputs.isotropic_mixture(n, d, 3, seed=n + d)
    sigma = float(np.sqrt(10.0 * d))
    param = {"gaussian": 2 * sigma * sigma, "laplacian": sigma}.get(kernel, 1.0)
    kind = {"gaussian": oracle.GAUSSIAN, "laplacian": oracle.LAPLACIAN, "linear": oracle.LINEAR,
            "poly": oracle.POLY}[kernel]
    k = min(n, 6)
    ref = oracle.kmeanspp(X.astype(np.float64), k, oracle.Kernel(kind, param, 1.0, 2), seed=3)
    Xd = torch.zeros(n, d + pad, device="cuda")
    Xd[:, :d] = torch.from_numpy(X).cuda()
    np.testing.assert_array_equal(kmeanspp(Xd[:, :d], k, kernel, param, coef0=1.0, degree=2, seed=3), ref)
