"""A call that steps queues all of its work before it returns: nothing is left
for kkm_flush, and the norms in a state read straight after it are those of the
step, whichever call took it."""
import numpy as np
import pytest

from paper_2410_05902_gb300 import inputs

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("precision,tile", [("bf16", 0), ("bf16", 64), ("tf32", 128), ("fp32", 0)])
def test_nothing_left_to_flush(precision, tile, graph):
    torch = torch_cuda()
    from paper_2410_05902_gb300.kkm import KKM
    n, d, k, b = 2000, 24, 8, 256
    X, _ = inputs.isotropic_mixture(n, d, k, seed=31)
    Xd = torch.from_numpy(X).cuda()
    run = KKM(Xd, k, b, kernel="gaussian", param=4.0 * d, tau=80, precision=precision, dist_tile=tile, seed=9,
              init_idx=inputs.init_indices(n, k, seed=32))
    run.graph(graph)
    batches = np.stack(inputs.batch_stream(n, b, 40, seed=35)).astype(np.int32)
    dev = torch.from_numpy(batches).cuda()
    calls = [lambda: run.step(dev[0]), lambda: run.step(), lambda: run.steps(1), lambda: run.steps(5),
             lambda: run.steps(16), lambda: run.steps(40), lambda: run.step_host(batches[1]),
             lambda: run.steps_host(batches), lambda: run.steps_host(batches[:7]), lambda: run.step_eval(dev[2])]
    steps = 0
    for _ in range(2):                       # the second time round on captured graphs
        for i, call in enumerate(calls):
            run.launches(reset=True)
            call()
            assert run.launches(reset=True) > 0
            run.flush()
            assert run.launches(reset=True) == 0, i
    run.sync()
    st = run.get_state()
    idx, w = torch.from_numpy(st["row_idx"]).cuda(), torch.from_numpy(st["row_w"]).cuda()
    ends = np.cumsum(st["rows_per_center"])
    tol = {"fp32": 1e-5, "tf32": 1e-2, "bf16": 5e-2}[precision]   # recurrence errors of a few dozen steps
    for j in range(k):
        sl = slice(int(ends[j] - st["rows_per_center"][j]), int(ends[j]))
        Y = Xd[idx[sl]].double()
        G = torch.exp(-torch.cdist(Y, Y).square() / (4.0 * d))
        assert abs(float(w[sl] @ G @ w[sl]) - st["cnorm"][j]) <= tol
    run.close()
