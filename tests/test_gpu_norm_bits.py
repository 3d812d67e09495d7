"""Bits of the center norms, on data whose exact sums need all of FP64's 53 bits
and where every FP32 step before them is exact."""
import numpy as np
import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["gaussian", "laplacian"])
@pytest.mark.parametrize("precision", ["fp32", "bf16", "bf16x3", "tf32"])
def test_window_sums_hold_fp64(precision, kernel):
    """One step of a run whose rows are all at the origin (every kernel value is
    1), with weights that are integers of up to 19 bits: a sum of 32 of them fits
    FP32, and A = sum_{D, W} w_p w_q and Bdd = sum_{D, D} w_p w_q fit 53 bits but
    not 48. The learning rate is so small that ||C'||^2 = ||C||^2 - 2 A + Bdd, from
    ||C||^2 = 0, is exact in FP64, to the last bit."""
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import KKM
    n, d, old, keep, b, tau = 400, 8, 100, 90, 120, 150
    X = torch.zeros(n, d, device="cuda")
    m = np.random.default_rng(3).integers(1 << 17, 1 << 19, size=old + keep) | 1
    run = KKM(X, 1, b, kernel=kernel, param=1.0, tau=tau, lr="const", eta=1e-300, precision=precision, seed=1,
              init_idx=np.zeros(1, np.int64))
    run.set_state(dict(iteration=3, rows_per_center=np.array([old + keep], np.int32),
                       row_idx=np.arange(old + keep, dtype=np.int64), row_w=m * 2.0 ** -19,
                       blocks_per_center=np.array([2], np.int32), block_iter=np.array([1, 2]),
                       block_count=np.array([old, keep], np.int32), c1_kept=np.zeros(1, np.uint8),
                       cnorm=np.zeros(1)))
    run.step(torch.arange(old + keep, old + keep + b, dtype=torch.int32, device="cuda"))
    st = run.get_state()
    assert st["rows_per_center"][0] == keep + b            # the older block left the window
    ints = [int(v) for v in m]
    a, bdd = sum(ints[:old]) * sum(ints), sum(ints[:old]) ** 2
    assert max(2 * a, a + bdd) < 1 << 53 and a > 1 << 49
    assert st["cnorm"][0] == float(bdd - 2 * a) * 2.0 ** -38
    run.close()
