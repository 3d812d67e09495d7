"""Steps in which one center takes 90 % of the batch: its window items number in
the hundreds, so its norm is the sum of several segments finished by different
CTAs, and its window is compacted while window items are in flight. Against the
FP64 oracle, and bit for bit between a run's own steps (singly, chained, through
host buffers) and the same run inside a group."""
import numpy as np
import pytest

from paper_2410_05902_gb300 import inputs

from gpu_helpers import CN_RTOL, DIST_TOL, OBJ_TOL_FORM, Pair, compare_states, dist_rel_err, torch_cuda

pytestmark = pytest.mark.gpu

N, D, K, B, TAU = 6000, 24, 6, 1500, 100


def _data():
    rng = np.random.default_rng(17)
    means = 3.0 * rng.normal(size=(K, D))
    lab = np.where(rng.random(N) < 0.9, 0, rng.integers(1, K, size=N))
    lab[:K] = np.arange(K)
    return (means[lab] + rng.normal(size=(N, D))).astype(np.float32)


@pytest.mark.parametrize("precision", ["fp32", "bf16x3", "bf16", "tf32"])
def test_forced_run_matches_oracle(precision):
    """Eight steps without a state reload, each with the oracle's assignment.
    A norm error of one step decays with (1 - alpha)^2 <= 0.74 (30 or more of
    1500 points to every center), so at most four one-step errors add up."""
    X = _data()
    p = Pair(X, k=K, b=B, tau=TAU, precision=precision, init=np.arange(K))
    most = 0
    for batch in inputs.batch_stream(N, B, 8, seed=5):
        rec = p.ora.step(batch)
        counts = np.bincount(rec.assign, minlength=K)
        assert counts.min() >= 15 and counts.max() > 1200
        most += counts.max()
        d, a, f = p.gpu_step(batch, forced=rec.assign)
        assert dist_rel_err(d, rec.dist) <= 4 * DIST_TOL[precision]
        assert abs(f - rec.batch_objective) <= 4 * OBJ_TOL_FORM[precision] * abs(rec.batch_objective)
    assert most > 2 * TAU + 4 * B + 8                  # the region was compacted on the way
    compare_states(p.gpu.get_state(), p.ora.state(), cn_rtol=4 * CN_RTOL[precision])
    p.close()


@pytest.mark.parametrize("kernel", ["gaussian", "linear"])
@pytest.mark.parametrize("precision,tile", [("fp32", 0), ("bf16x3", 0), ("bf16", 0), ("bf16", 64), ("tf32", 128)])
def test_ways_to_step_agree(precision, tile, kernel):
    torch = torch_cuda()
    from paper_2410_05902_gb300.group import Group
    from paper_2410_05902_gb300.kkm import KKM
    Xd = torch.from_numpy(_data()).cuda()
    runs = [KKM(Xd, K, B, kernel=kernel, param=4.0 * D, tau=TAU, precision=precision, dist_tile=tile, seed=9,
                init_idx=np.arange(K, dtype=np.int64)) for _ in range(4)]
    single, chain, host, grouped = runs
    for r in runs:
        r.graph(True)
    g = Group([grouped])
    for _ in range(21):
        single.step()
        g.step()
    g.sync()
    chain.steps(21)
    host.steps_host(None, n=21)
    want = single.get_state()
    assert np.max(want["rows_per_center"]) > (1000 if kernel == "gaussian" else 0)
    for r in (chain, host, grouped):
        got = r.get_state()
        for key in want:
            assert np.array_equal(np.asarray(got[key]), np.asarray(want[key])), key
    for r in runs:
        r.close()
