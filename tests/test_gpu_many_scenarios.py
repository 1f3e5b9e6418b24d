"""Scenario counts beyond what a tensor map's coordinates reach: the rollouts take
the per-lane ring there, on batched and on single handles, with the draws of
every scenario."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).total_memory < 120e9:
        pytest.skip("needs 120 GB of device memory")
    from paper_2510_08288_gb300 import build as B
    B.build()
    from paper_2510_08288_gb300 import rrg
    return rrg


def test_batch_of_more_than_2_30_scenarios(R, orc, params):
    """Counts whose tensor map the driver refuses (dimensions end at 2^32
    elements, four a scenario) are accepted, and the update runs."""
    cfg = R.rrg_config_default(max_candidates=1, search=R.SEARCH_SPEC_BISECT, precision=R.FP32_RECHECK, n_bisect=1)
    x = orc.equilibrium(params, 100.0)
    with R.BatchGovernor(params, cfg, [2 ** 30 + 4], [1]) as g:
        v, kappa, flags = g.step(x, [100.0], [100.0], 1, 0)
        assert (v[0], kappa[0], flags[0]) == (100.0, 1.0, 0)
        st = g.stats()
        assert st["lane_steps"] == 2 ** 30 + 4 and st["wait_timeouts"] == 0
