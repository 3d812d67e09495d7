"""A hand-over whose wait runs out leaves the slot's value and its reader's
barrier untouched (kkm_probe_bounded_wait with nothing arriving reports a state
error when it does not), and one that is let through delivers."""
import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit_ns", [1000, 300_000])
def test_hand_over_gives_up_without_a_trace(limit_ns):
    import time
    torch = torch_cuda()
    from paper_2410_05902_gb300 import kkm
    stream = torch.cuda.current_stream().cuda_stream
    kkm.kkm_probe_bounded_wait(limit_ns, True, stream)
    t0 = time.perf_counter()
    assert kkm.kkm_probe_bounded_wait(limit_ns, False, stream) == kkm.KKM_ETIMEOUT
    assert time.perf_counter() - t0 >= 2e-9 * limit_ns         # the wait and the hand-over's
    assert kkm.kkm_probe_bounded_wait(limit_ns, True, stream) == kkm.KKM_OK
