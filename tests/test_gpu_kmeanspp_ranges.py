"""Kernel k-means++ at the edges of its draw kernel: blocks of 128 points with
remainders, feature tiles of 32 with remainders, rows that cannot be read 16
bytes at a time, and values whose squares leave FP32's range (where the FP32
triples give way to FP64). The chosen indices must equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2410_05902_gb300 import inputs

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,n,d,pad,k,scale", [
    ("gaussian", 129, 33, 0, 8, 1.0),
    ("gaussian", 128, 32, 0, 8, 1.0),
    ("laplacian", 1000, 300, 0, 9, 1.0),
    ("gaussian", 700, 36, 4, 9, 1.0),       # strided rows, 16-byte loads
    ("gaussian", 700, 36, 3, 9, 1.0),       # strided rows, scalar loads
    ("poly", 300, 65, 1, 6, 1.0),
    ("linear", 257, 31, 0, 6, 1.0),
    ("gaussian", 400, 40, 0, 8, 1e-22),     # squares below FP32's range
    ("gaussian", 400, 40, 0, 8, 1e19),      # squares above it
    ("gaussian", 1, 4, 0, 1, 1.0),
])
def test_kmeanspp_edges(kernel, n, d, pad, k, scale):
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import kmeanspp
    X, _ = inputs.isotropic_mixture(max(n, 2), d, 4, seed=n + d)
    X = (X[:n].astype(np.float64) * scale).astype(np.float32)
    sigma = scale * float(np.sqrt(10.0 * d))
    param = {"gaussian": 2 * sigma * sigma, "laplacian": sigma}.get(kernel, 1.0)
    kind = {"gaussian": oracle.GAUSSIAN, "laplacian": oracle.LAPLACIAN, "linear": oracle.LINEAR,
            "poly": oracle.POLY}[kernel]
    ref = oracle.kmeanspp(X.astype(np.float64), k, oracle.Kernel(kind, param, 1.0, 2), seed=3)
    Xd = torch.zeros(n, d + pad, device="cuda")
    Xd[:, :d] = torch.from_numpy(X).cuda()
    got = kmeanspp(Xd[:, :d], k, kernel, param, coef0=1.0, degree=2, seed=3)
    np.testing.assert_array_equal(got, ref)
