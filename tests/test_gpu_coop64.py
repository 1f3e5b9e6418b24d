"""Four lanes per binary64 trajectory (small binary64 launches) against one lane
per trajectory: lanes that draw their disturbances in the trajectory loop, and
launches with too many candidates for the split.  The arithmetic is the same
operation by operation, so the results are equal."""
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


@pytest.mark.parametrize("H", [1, 3, 4, 5, 8, 50])
@pytest.mark.parametrize("N", [1, 7, 8, 9, 33, 257])
@pytest.mark.parametrize("unc", [0.0, 0.1])
@pytest.mark.parametrize("early_exit", [0, 1])
def test_equals_one_lane_per_trajectory(R, params, H, N, unc, early_exit):
    kap = np.array([0.0, 0.05, 0.3, 1.0])
    out = []
    for gen in (1, 0):
        cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=4, precision=R.FP64,
                                   early_exit=early_exit, scenarios_in_register=gen, param_unc_rel=unc)
        with R.Governor(params, cfg) as g:
            x, _ = g.equilibrium(100.0)
            g.sample_scenarios(5, 9)
            # the second target takes the compressor's pressure ratio off the power's table
            out.append([g.eval_candidates(x, 100.0, r, kap, want_P=True) for r in (160.0, 2000.0)])
    for a, b in zip(out[0], out[1]):
        for u, v in zip(a, b):
            if early_exit == 0 or u.dtype != np.float64:
                np.testing.assert_array_equal(u, v)


@pytest.mark.parametrize("probe", [1, 4, 6, 13])
@pytest.mark.parametrize("N", [5, 64])
def test_segments_equal_one_lane_per_trajectory(R, params, probe, N):
    got = []
    for gen in (1, 0):
        cfg = R.rrg_config_default(horizon=70, n_scenarios=N, max_candidates=15, probe_steps=probe,
                                   precision=R.FP64, scenarios_in_register=gen)
        with R.Governor(params, cfg) as g:
            x, _ = g.equilibrium(100.0)
            for t in range(3):
                g.sample_scenarios(t, 4)
                got.append(g.step(x * (1.0 + 0.004 * t), 230.0, 100.0)[1:])
    assert got[:3] == got[3:]


@pytest.mark.parametrize("H,checkpoint", [(1, 1), (5, 2), (60, 50)])
@pytest.mark.parametrize("unc", [0.0, 0.1])
def test_gradient_equals_one_lane_per_trajectory(R, params, H, checkpoint, unc):
    """One call for 24 kappas takes one lane per trajectory, calls for three of
    them take four."""
    kap = np.linspace(0.0, 1.0, 24)
    with R.Governor(params, R.rrg_config_default(horizon=H, n_scenarios=997, max_candidates=24,
                                                 param_unc_rel=unc)) as g:
        x, _ = g.equilibrium(100.0)
        g.sample_scenarios(2, 1)
        a = g.slack_gradients(x, 100.0, 200.0, kap, checkpoint, R.FP64)
        for i in range(0, 24, 3):
            b = g.slack_gradients(x, 100.0, 200.0, kap[i:i + 3], checkpoint, R.FP64)
            for u, v in zip(a, b):
                np.testing.assert_array_equal(u[i:i + 3], v)
