"""Distance passes on CTA pairs with 128-column tiles, many items to a pair: two
items share a pass over their row tile, the accumulators and the metadata slots
of both CTAs go round many times, descriptors are fetched anew after every 32
items, and every group takes items of its own. Odd numbers of row tiles, ragged
last ones, and queries that are no support rows (so that the Laplacian's
distances can be held to the oracle)."""
import numpy as np
import pytest

import oracle
from paper_2410_05902_gb300 import inputs

from gpu_helpers import DIST_TOL, KIND, Pair, dist_rel_err, torch_cuda

pytestmark = pytest.mark.gpu


def _sms(torch):
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("kernel", ["gaussian", "laplacian"])
@pytest.mark.parametrize("precision,d", [("bf16", 400), ("bf16x3", 200), ("tf32", 230)])
def test_windows_many_items_per_pair(precision, d, kernel):
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import KKM
    n, k, b, tau = 20_000, 96, 2817, 300          # 23 row tiles, the last of one row
    X, _ = inputs.isotropic_mixture(n + b, d, k, seed=d)
    X, Q = X[:n], X[n:]
    sigma = inputs.median_sigma(X, seed=1)
    param = 2 * sigma * sigma if kernel == "gaussian" else sigma
    run = KKM(torch.from_numpy(X).cuda(), k, b, kernel=kernel, param=param, tau=tau, precision=precision,
              dist_tile=128, seed=2, init_idx=inputs.init_indices(n, k, seed=3))
    run.steps(14)
    st = run.get_state()
    rows = st["rows_per_center"].astype(np.int64)
    pick = np.random.default_rng(1).choice(b, size=48, replace=False)
    pick[:3] = (0, 2815, 2816)
    kern = oracle.Kernel(KIND[kernel], param)
    ref, st["cnorm"] = oracle.state_distances(X.astype(np.float64), Q[pick].astype(np.float64), st, kern)
    run.set_state(st)            # exact norms: the distances' own error is what is left
    tiles, R = int(np.sum((rows + 127) // 128)), (b + 127) // 128
    sms = _sms(torch)
    assert R % 2 == 1 and (R + 1) // 2 * tiles > 32 * (sms // 2)     # more than one fetch of 32 descriptors a pair
    assert 3 * tiles >= 4 * sms                                  # three row tiles: teams too, but no pairs
    Qd = torch.from_numpy(Q).cuda()
    _, _, dist = run.assign(Qd, want_dist=True)
    got = dist.cpu().numpy()
    err = float(np.max(np.abs(got[pick].astype(np.float64) - ref)) / np.max(np.abs(ref)))
    assert err <= DIST_TOL[precision], f"normwise distance error {err:.3e}"
    for s in range(0, b, 384):   # bit for bit what single CTAs give the same rows
        m = min(384, b - s)
        if 3 * 128 - m >= 128:
            s, m = b - 384, 384  # (the last rows once more, in three full row tiles)
        _, _, part = run.assign(Qd[s:s + m].contiguous(), want_dist=True)
        np.testing.assert_array_equal(got[s:s + m], part.cpu().numpy())
    run.close()


@pytest.mark.parametrize("precision,d", [("bf16", 450), ("bf16x3", 200), ("tf32", 230)])
def test_table_many_items_per_pair(precision, d):
    """The table form's default tiles of wide rows: every row of X against the
    batch's blocks, 547 row tiles."""
    torch = torch_cuda()
    n, k, b = 69_930, 5, 1024
    X, _ = inputs.isotropic_mixture(n, d, k, seed=12)
    R = (n + 127) // 128
    assert R % 2 == 1
    p = Pair(X, k=k, b=b, tau=0, precision=precision, algo="table")
    rng = np.random.default_rng(6)
    for i in range(3):
        B = rng.choice(n, size=b)
        B[:4] = (0, n - 1, n - 2, n - 130)        # the first row, the ragged last row tile
        rec = p.ora.step(B)
        tiles = int(np.sum((np.bincount(rec.assign, minlength=k) + 127) // 128))
        assert (R + 1) // 2 * tiles > 32 * (_sms(torch) // 2)
        dist, _, _ = p.gpu_step(B, forced=rec.assign)
        assert dist_rel_err(dist, rec.dist) <= DIST_TOL[precision], i
    p.close()
