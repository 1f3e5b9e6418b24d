"""Binary64 handles whose scenarios have exponents of their own (gamma uncertain, or
explicit multipliers of it): the power table does not hold them, so four lanes per
trajectory pay only while a scheduler has one warp.  Results equal between the forms,
and two warps a scheduler are not slower than twice as many trajectories."""
import numpy as np
import pytest

from paper_2510_08288_gb300 import inputs

pytestmark = pytest.mark.gpu

GAMMA = inputs.FC3_PARAM_NAMES.index("gamma")


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_08288_gb300 import build as B
    B.build()
    from paper_2510_08288_gb300 import rrg
    return rrg


def _cfg(R, N, m, **kw):
    base = dict(horizon=50, n_scenarios=N, max_candidates=m, precision=R.FP64, early_exit=R.EXIT_NONE,
                param_unc_rel=0.05, param_unc_mask=inputs.FC3_UNCERTAIN_MASK | 1 << GAMMA)
    base.update(kw)
    return R.rrg_config_default(**base)


@pytest.mark.parametrize("explicit", [False, True])
def test_forms_give_the_same_results(R, params, explicit):
    """8, 600 (four lanes), 1,100 and 2,048 (one lane) scenarios: the first ones agree."""
    k = np.linspace(0.0, 0.6, 8)
    out = []
    for N in (8, 600, 1100, 2048):
        kw = dict(param_unc_mask=inputs.FC3_UNCERTAIN_MASK) if explicit else {}
        with R.Governor(params, _cfg(R, N, 8, y_min=2.0, **kw)) as g:
            x, _ = g.equilibrium(100.0)
            g.sample_scenarios(1, 0)
            if explicit:
                m = g.get_param_multipliers()
                m[:, GAMMA] = 1.0 + 0.01 * np.cos(np.arange(N))
                g.set_param_multipliers(m)
            out.append(g.eval_candidates(x, 100.0, 250.0, k, want_P=True)[2][:, :8])
            grad = [g.slack_gradients(x, 100.0, 250.0, k[1:3])[0]]
    assert 0 < out[0].sum() < out[0].size
    for P in out[1:]:
        np.testing.assert_array_equal(P, out[0])
    assert np.all(np.isfinite(grad))


@pytest.mark.parametrize("explicit", [False, True])
def test_two_warps_a_scheduler_are_not_slower(R, params, explicit):
    k = np.linspace(0.0, 0.05, 8)
    ms = []
    for N in (1024, 2048):
        kw = dict(param_unc_mask=inputs.FC3_UNCERTAIN_MASK) if explicit else {}
        with R.Governor(params, _cfg(R, N, 8, **kw)) as g:
            x, _ = g.equilibrium(100.0)
            g.sample_scenarios(1, 0)
            if explicit:
                m = g.get_param_multipliers()
                m[:, GAMMA] = 1.01
                g.set_param_multipliers(m)
            g.set_profiling(True)
            g.eval_candidates(x, 100.0, 150.0, k)
            g.reset_stats()
            for _ in range(5):
                g.eval_candidates(x, 100.0, 150.0, k)
            st = g.stats()
            ms.append(st["rollout_ms"] / st["timed_rollouts"])
    print("1,024 and 2,048 scenarios x 8:", ms)
    assert ms[0] < 1.25 * ms[1]
