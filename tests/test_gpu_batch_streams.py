"""The batched handle's work stays on its own stream."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_08288_gb300 import build as B
    B.build()
    from paper_2510_08288_gb300 import rrg
    return rrg


def test_first_closed_loop_call_is_ordered_on_the_handles_stream(R, params):
    """The first closed-loop call, which sets up the second scenario pair and its
    tensor maps, leaves the legacy stream alone: it returns while that stream is
    busy (what it copies there would not be ordered before the handle's kernels)."""
    import torch
    cfg = R.rrg_config_default(max_candidates=2, search=R.SEARCH_KSECTION, precision=R.FP32_RECHECK)
    r = torch.full((1,), 150.0, dtype=torch.float64, device="cuda")
    with R.BatchGovernor(params, cfg, [64], [32]) as g:
        torch.cuda.synchronize()
        busy = torch.cuda.Event()
        torch.cuda._sleep(1 << 30)
        busy.record()
        R.rrg_batch_closed_loop_dev(g.h, None, None, r, 0, 1, 0, np.zeros(3), False)
        assert not busy.query()
        torch.cuda.synchronize()
