"""Distance passes whose operands stream (wide rows): CTA pairs on two row tiles.

Sizes where the pairing can go wrong: an odd last row tile (the pair's second
CTA has no rows), a ragged last row tile, support tiles of a few columns, of
just over half and of all 256, one slice short of and past a ring of stages,
and batches too small to pair. Distances against the FP64 oracle, held to each
form's bound, and bit for bit against the same rows scored without a pair.
"""
import numpy as np
import pytest

import oracle
from paper_2410_05902_gb300 import inputs

from gpu_helpers import DIST_TOL, KIND, Pair, dist_rel_err, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["gaussian", "laplacian", "linear"])
@pytest.mark.parametrize("precision,d,tile", [
    ("bf16", 300, 128), ("bf16", 784, 128), ("bf16x3", 129, 128), ("bf16x3", 257, 128), ("tf32", 129, 128),
    ("tf32", 230, 128), ("bf16", 1030, 256), ("bf16x3", 321, 256), ("tf32", 490, 256)])
def test_paired_row_tiles_match_oracle(kernel, precision, d, tile):
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import KKM
    n, k, b, tau = 3000, 5, 900, 260
    X, _ = inputs.isotropic_mixture(n, d, k, seed=d)
    sigma = inputs.median_sigma(X, seed=1)
    param = {"gaussian": 2 * sigma * sigma, "laplacian": sigma, "linear": 1.0}[kernel]
    run = KKM(torch.from_numpy(X).cuda(), k, b, kernel=kernel, param=param, tau=tau, precision=precision,
              dist_tile=tile, init_idx=inputs.init_indices(n, k, seed=3))
    for batch in inputs.batch_stream(n, b, 3, seed=4):
        run.step(torch.from_numpy(batch.astype(np.int32)).cuda())
    st = run.get_state()
    kern = oracle.Kernel(KIND[kernel], param)
    Q = X[:b]
    ref, st["cnorm"] = oracle.state_distances(X.astype(np.float64), Q.astype(np.float64), st, kern)
    run.set_state(st)            # exact norms: the distances' own error is what is left
    scale = float(np.max(np.abs(ref)))
    out = {}
    for m in (1, 128, 129, 256, 384, 513, 640, 897, 900):   # 1 to 8 row tiles, odd and ragged counts
        _, _, dist = run.assign(torch.from_numpy(Q[:m]).cuda(), want_dist=True)
        out[m] = dist.cpu().numpy()
        # the Laplacian's square root magnifies the cancellation of a query that equals a
        # support row (kkm_assign knows no indices for query rows), so its values are held
        # to the unpaired ones only
        err = float(np.max(np.abs(out[m].astype(np.float64) - ref[:m]))) / scale
        assert kernel == "laplacian" or err <= DIST_TOL[precision], f"m = {m}: normwise distance error {err:.3e}"
    for m in out:                # alone or in a pair, a row's distances are the same bits
        np.testing.assert_array_equal(out[m], out[900][:m])
    run.close()


@pytest.mark.parametrize("counts", ["even", "skewed"])
def test_table_blocks_of_wide_rows_match_oracle(counts):
    n, d, k, b = 1500, 450, 4, 700
    X, labels = inputs.isotropic_mixture(n, d, k, seed=11)
    p = Pair(X, k=k, b=b, tau=0, precision="bf16", algo="table")
    rng = np.random.default_rng(5)
    pool = np.arange(n) if counts == "even" else np.nonzero(labels == labels[0])[0]   # skewed: one block of all rows
    for _ in range(3):
        B = rng.choice(pool, size=b)
        rec = p.ora.step(B)
        dist, _, _ = p.gpu_step(B, forced=rec.assign)
        assert dist_rel_err(dist, rec.dist) <= DIST_TOL["bf16"]
    p.close()


def test_paired_table_steps_replayed_from_a_graph():
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import KKM
    X, _ = inputs.isotropic_mixture(1500, 450, 4, seed=13)
    sigma = inputs.median_sigma(X, seed=1)
    out = []
    for graph in (False, True):
        run = KKM(torch.from_numpy(X).cuda(), 4, 300, kernel="gaussian", param=2 * sigma * sigma, tau=0, algo="table",
                  precision="bf16", seed=3, init_idx=inputs.init_indices(len(X), 4, seed=3))
        run.graph(graph)
        run.steps(40)            # eager steps and two replays of sixteen, or forty eager ones
        dist = torch.empty((300, 4), dtype=torch.float32, device="cuda")
        run.step(torch.arange(300, dtype=torch.int32, device="cuda"), None, None, dist, None)
        out.append((dist.cpu().numpy(), run.objective()))
        run.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
