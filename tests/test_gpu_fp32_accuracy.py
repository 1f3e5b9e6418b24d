"""The size of the binary32 rollouts' error against binary64: no larger than that
of the step with its right-hand sides evaluated stage by stage, whose figures on
these updates (measured on a GB300 before the linear part was folded) are the
bounds: the median trajectory's and the largest error of a trajectory's slacks."""
import numpy as np
import pytest

from paper_2510_08288_gb300 import inputs

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


@pytest.mark.parametrize("N,H,M,unc,start,updates,median,largest", [
    (1024, 2000, 16, 0.0, "equilibrium", 12, 2.012e-7, 3.17e-6),
    (512, 3000, 16, 0.0, "far", 12, 2.620e-7, 6.25e-6),
    (1024, 2000, 16, 0.1, "near", 8, 2.244e-7, 6.14e-6),
    (64, 300, 8, 0.0, "near", 24, 1.995e-7, 5.00e-6),
])
def test_error_no_larger_than_stage_by_stage(R, params, N, H, M, unc, start, updates, median, largest):
    rng = np.random.default_rng(7)
    med, big = [], 0.0
    with R.Governor(params, R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=M, precision=R.FP32_RECHECK,
                                                 recheck_eps_rel=1e-6, param_unc_rel=unc,
                                                 param_unc_mask=inputs.FC3_UNCERTAIN_MASK)) as g:
        for t in range(updates):
            v, r = rng.uniform(50, 300, 2)
            x, _ = g.equilibrium(v)
            if start == "near":
                x = x + np.array([150.0, 20.0, 150.0]) * rng.uniform(-1, 1, 3)
            elif start == "far":
                x = x * rng.uniform(0.9, 1.1, 3)
            g.sample_scenarios(11, t)
            err = g.slack_error(x, v, r, np.linspace(0, 1, M))["err"]
            med.append(np.median(err))
            big = max(big, float(err.max()))
    print("median %.3e (bound %.3e), largest %.3e (bound %.3e)" % (np.mean(med), median, big, largest))
    assert np.mean(med) <= median and big <= largest
