"""Bits of the allocation-free call's row norms: FP64 sums rounded once to FP32."""
import numpy as np
import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [4, 5, 300])
def test_row_norms_round_as_fp64_sums(d):
    """||q||^2 of rows whose sum of squares lies 2^-52 above the midpoint of two
    FP32 values: the norm is FP64's sum rounded once, so the upper one. With the
    linear kernel and no support rows the distance is the norm."""
    torch = torch_cuda()
    from paper_2410_05902_gb300 import kkm as K
    m = 70
    Q = torch.zeros(m, d, device="cuda")
    rng = np.random.default_rng(d)
    for r in range(m):
        at = rng.choice(d, size=3, replace=False)
        Q[r, at[0]], Q[r, at[1]] = 1.0, 2.0 ** -12
        Q[r, at[2]] = 2.0 ** -26 if r % 2 else 0.0
    out = torch.empty(m, 1, device="cuda")
    off, cn = torch.zeros(2, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    kern = K.kkm_kernel(K.KKM_LINEAR, 1.0, 0.0, 1)
    K.kkm_distances_noalloc(Q.data_ptr(), m, d, d, None, 0, d, None, off.data_ptr(), cn.data_ptr(), 1, kern,
                            out.data_ptr(), None, torch.cuda.current_stream().cuda_stream)
    want = [1.0 + 2.0 ** -23 if r % 2 else 1.0 for r in range(m)]   # without the third: the midpoint, to even
    np.testing.assert_array_equal(out.cpu().numpy()[:, 0], np.array(want, np.float32))
