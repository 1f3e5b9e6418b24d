"""The reverse sweep's chunks of 32 steps and its checkpoint segments, around
their edges: a disturbance puts the least slack at a chosen step."""
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


@pytest.mark.parametrize("jstar", [1, 2, 31, 32, 33, 64, 65, 100])
@pytest.mark.parametrize("checkpoint", [1, 16, 30, 200])
@pytest.mark.parametrize("unc", [0.0, 0.1])
def test_sweep_from_any_step(R, orc, params, jstar, checkpoint, unc):
    """FP64 against the oracle's complex-step gradient (1e-7, as everywhere for
    it); FP32 against FP64 to 1e-3 of the largest entry per group."""
    N, H, v_prev, r, kappa = 9, 100, 100.0, 130.0, 0.2
    x_t = orc.equilibrium(params, v_prev)
    d = orc.sample_disturbances(3, 1, N, H, inputs.DIST_AMP).reshape(3, H, N)
    d[2, jstar - 1, 4] -= 60.0 * inputs.DIST_AMP[2]
    with R.Governor(params, R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=2, param_unc_rel=unc)) as g:
        g.sample_scenarios(3, 1)
        m = g.get_param_multipliers() if unc else None
        g.set_scenarios(d)
        gv, grad, ks, js = g.slack_gradient(x_t, v_prev, r, kappa, checkpoint, R.FP64)
        g32, grad32, k32, j32 = g.slack_gradient(x_t, v_prev, r, kappa, checkpoint, R.FP32)
    assert (ks, js) == (4, jstar) == (k32, j32)
    with orc.param_multipliers(m):
        s, gro = orc.slack_grad(params, orc.cfg(H=H, N=N, early_exit=0), x_t, v_prev, r, kappa, d, 4, jstar)
    assert gv == pytest.approx(s, rel=1e-10, abs=1e-12)
    np.testing.assert_allclose(grad, gro, rtol=1e-7, atol=1e-14 * np.max(np.abs(gro)))
    for sl in (slice(0, 1), slice(1, 4), slice(4, 31)):
        assert np.all(np.abs(grad32[sl] - grad[sl]) <= 1e-3 * np.max(np.abs(grad[sl])))
