"""The rollout step whose linear part is folded through the RK4 stages, at the
places where its pieces change: the cells and the ends of the binary64 x^e - 1
table and exponents it does not cover, and the scenarios' models folded with
the draw (parametric uncertainty) at warp remainders and for loaded
multipliers."""
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


@pytest.mark.parametrize("gamma", [1.4, 1.05, 2.0, 0.4])
@pytest.mark.parametrize("x_sm", [1.0, 1.0 + 2.0 ** -9, 1.2, 1.999, 2.0, 2.4])
def test_binary64_power_table_cells_and_ends(R, orc, gamma, x_sm):
    """x = p_sm / p_atm at the table's first cell, a cell's edge, inside, its
    last cell and beyond it (the fall-back to pow), for exponents (gamma - 1) /
    gamma inside [-1, 1] and, at gamma = 0.4, outside: three steps of the
    binary64 rollout against the oracle (both round each operation in binary64,
    so a few hundred operations of relative error 1.1e-16 on slacks of order 1
    to 100 stay below 1e-11 of the largest)."""
    p = inputs.fc3_params(gamma=gamma)
    N, H = 5, 3
    d = inputs.uniform_disturbances(N, H, 3)
    x_t = np.array([x_sm * 101325.0 - 8000.0, 3300.0, x_sm * 101325.0])
    kap = np.array([0.0, 0.4, 1.0])
    cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=4, precision=R.FP64, early_exit=0, ss_check=0)
    with R.Governor(p, cfg) as g:
        g.set_scenarios(d)
        _, ms, P = g.eval_candidates(x_t, 100.0, 180.0, kap, want_P=True)
    c = orc.cfg(H=H, N=N, early_exit=0, ss_check=0)
    _, mo, Po, _ = orc.eval_candidates(p, c, x_t, 100.0, 180.0, kap, d, want_P=True)
    np.testing.assert_allclose(ms, mo, rtol=1e-11, atol=1e-11)
    np.testing.assert_array_equal(P, Po)


@pytest.mark.parametrize("N", [1, 31, 33, 130])
@pytest.mark.parametrize("tma", [0, 2])
def test_folded_scenario_models_match_binary64(R, N, tma):
    """Parametric uncertainty, drawn and loaded multipliers: the binary32 lanes
    read their scenario's model from the arrays folded after the draw, the
    binary64 lanes fold it themselves.  Their min slacks agree to the binary32
    error of the power term, about 6e-8 x 0.3 / 0.06 of a slack of order 1 per
    stage, below 1e-5 after the step's contraction."""
    H, M = 40, 5
    p = inputs.fc3_params()
    kap = np.linspace(0.0, 0.3, M)
    out = {}
    for prec in (R.FP32, R.FP64):
        cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=8, precision=prec, early_exit=0,
                                   param_unc_rel=0.1)
        with R.Governor(p, cfg) as g:
            if g.get_tma() != R.TMA_NEVER:
                g.set_tma(tma)
            x, _ = g.equilibrium(120.0)
            g.sample_scenarios(11, 3)
            a = g.eval_candidates(x, 120.0, 200.0, kap)[1]
            m = np.random.default_rng(5).uniform(0.93, 1.07, size=(N, R.NPARAM))
            m[:, 22:] = 1.0
            m[:, 0] = 1.0  # p_atm shifts the start by its whole change
            g.set_param_multipliers(m)
            b = g.eval_candidates(x, 120.0, 200.0, kap)[1]
            out[prec] = (a, b)
    for a, b in zip(out[R.FP32], out[R.FP64]):
        assert np.array_equal(np.isnan(a), np.isnan(b))
        ok = ~np.isnan(a)
        assert ok.any()
        assert np.max(np.abs(a[ok] - b[ok])) < 1e-5
