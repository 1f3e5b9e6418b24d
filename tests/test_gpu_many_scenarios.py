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


N_BIG, TAIL = 2 ** 29 + 64, 64


def _boundary(R, orc, params):
    """A state one step of which the disturbances decide: y_min is the output
    that the undisturbed step reaches, just below the start's."""
    x = orc.equilibrium(params, 150.0)
    with R.Governor(params, R.rrg_config_default(horizon=1, n_scenarios=1, ss_check=0, y_min=1.0)) as g:
        _, slack, _ = g.eval_candidates(x, 150.0, 150.0, [0.0])  # no disturbance drawn: both outputs
    return x, 1.0 + float(slack[0]) - 1e-4


def test_single_handle_draws_past_scenario_2_29(R, orc, params):
    """Scenarios from 2^29 on have the admissibility of the same scenarios on a
    handle that holds only them: about half of them violate."""
    x, y_min = _boundary(R, orc, params)
    kw = dict(horizon=1, max_candidates=1, search=R.SEARCH_BISECT, precision=R.FP32, early_exit=R.EXIT_NONE,
              ss_check=0, y_min=y_min)
    with R.Governor(params, R.rrg_config_default(n_scenarios=TAIL, scenario_base=N_BIG - TAIL, **kw)) as g:
        g.sample_scenarios(3, 0)
        want = g.eval_candidates(x, 150.0, 150.0, [0.0], want_P=True)[2][0]
    assert 0 < want.sum() < TAIL
    with R.Governor(params, R.rrg_config_default(n_scenarios=N_BIG, **kw)) as g:
        assert g.get_tma() == R.TMA_NEVER
        g.sample_scenarios(3, 0)
        got = g.eval_candidates(x, 150.0, 150.0, [0.0], want_P=True)[2][0]
    np.testing.assert_array_equal(got[-TAIL:], want)
    assert 0.3 < got[:1 << 20].mean() < 0.7


def test_batch_draws_past_scenario_2_29(R, orc, params):
    """As many scenarios in a batch (ring of quads throughout), counted by the binary64 recheck: no slack is
    negative, and the band ends where an undisturbed step's slack lies, so the
    last 64 scenarios add as many rechecks as have a lower slack."""
    x, y_mid = _boundary(R, orc, params)
    eps = 0.02  # far above the slacks' spread, so none is negative
    y_min = y_mid / (1.0 + eps)  # y_min + eps y_min: just below the undisturbed output
    kw = dict(max_candidates=1, search=R.SEARCH_SPEC_BISECT, precision=R.FP32_RECHECK, n_bisect=1, ss_check=0,
              early_exit=R.EXIT_LANE)
    count = []
    for N in (2 ** 29, N_BIG):
        with R.BatchGovernor(params, R.rrg_config_default(y_min=y_min, recheck_eps_rel=eps, **kw), [N], [1]) as g:
            _, kappa, flags = g.step(x, [150.0], [150.0], 3, 0)
            assert (kappa[0], flags[0]) == (1.0, 0)
            count.append(g.stats()["rechecked"])
    kw.update(search=R.SEARCH_BISECT, precision=R.FP32, early_exit=R.EXIT_NONE, horizon=1)
    with R.Governor(params, R.rrg_config_default(y_min=y_mid, n_scenarios=TAIL, scenario_base=N_BIG - TAIL,
                                                 **kw)) as g:
        g.sample_scenarios(3, 0)
        above = g.eval_candidates(x, 150.0, 150.0, [0.0], want_P=True)[2][0]
    assert 0 < above.sum() < TAIL
    assert count[1] - count[0] == TAIL - int(above.sum())
