"""The quad layout of the binary32 scenario arrays (four steps of a scenario
side by side) at horizons around a quad, a block of quads and a TMA chunk: the
ring of quads and the TMA ring against lanes that draw their disturbances in the
trajectory loop, segments that start inside a quad, explicit scenarios, and the
gradient's forward pass and its saved states."""
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


HORIZONS = [1, 3, 4, 5, 15, 16, 17, 19, 20, 31, 33, 35, 64, 67]


@pytest.mark.parametrize("H", HORIZONS)
@pytest.mark.parametrize("N", [1, 33, 132])
@pytest.mark.parametrize("unc", [0.0, 0.1])
def test_rings_equal_the_draw_in_the_loop(R, params, H, N, unc):
    kap = np.array([0.0, 0.05, 0.3, 1.0])
    out = []
    for gen, tma in ((1, None), (0, 0), (0, 2)):
        cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=4, precision=R.FP32, early_exit=0,
                                   scenarios_in_register=gen, param_unc_rel=unc)
        with R.Governor(params, cfg) as g:
            if tma is not None and g.get_tma() != R.TMA_NEVER:
                g.set_tma(tma)
            x, _ = g.equilibrium(100.0)
            g.sample_scenarios(5, 9)
            out.append(g.eval_candidates(x, 100.0, 160.0, kap, want_P=True))
    for o in out[1:]:
        for a, b in zip(out[0], o):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("H", [5, 17, 70])
@pytest.mark.parametrize("probe", [1, 2, 3, 4, 6, 13])
@pytest.mark.parametrize("tma", [0, 2])
def test_segments_that_start_inside_a_quad(R, orc, params, H, probe, tma):
    """Continuations of a probe of any length give Alg. 1's kappa."""
    if probe >= H:
        pytest.skip("the probe covers the horizon")
    N = 64
    for seed in range(3):
        x = orc.equilibrium(params, 100.0) * (1.0 + 0.004 * seed)
        d = orc.sample_disturbances(seed, 4, N, H, inputs.DIST_AMP)
        cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=15, probe_steps=probe)
        with R.Governor(params, cfg) as g:
            g.set_tma(tma)
            g.sample_scenarios(seed, 4)
            _, k, f = g.step(x, 230.0, 100.0)
            # explicit scenarios: the binary64 draw, rounded into the layout
            g.set_scenarios(d)
            _, k2, f2 = g.step(x, 230.0, 100.0)
        ref = orc.bisect_joint(params, orc.cfg(H=H, N=N), x, 100.0, 230.0, 12, d)
        assert (k, f) == ref and (k2, f2) == ref


@pytest.mark.parametrize("H", [1, 2, 15, 16, 17, 33, 64, 100])
@pytest.mark.parametrize("checkpoint", [1, 15, 16, 17, 50])
def test_binary32_gradient_between_blocks(R, params, H, checkpoint):
    """The binary32 gradient against the binary64 one on the same draw: g to the
    binary32 slack error (below 1e-5, see the model's power term), the same
    argmin, and the gradient to 1e-3 of its largest entry per group (binary32
    products over at most 100 steps, each relative error 6e-8, times a
    condition below 100)."""
    N = 40
    with R.Governor(params, R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=4)) as g:
        x, _ = g.equilibrium(100.0)
        g.sample_scenarios(2, 1)
        kap = np.array([0.0, 0.2, 0.6])
        a = g.slack_gradients(x, 100.0, 200.0, kap, checkpoint, R.FP32)
        b = g.slack_gradients(x, 100.0, 200.0, kap, checkpoint, R.FP64)
    np.testing.assert_allclose(a[0], b[0], rtol=0, atol=1e-5)
    np.testing.assert_array_equal(a[2], b[2])
    np.testing.assert_array_equal(a[3], b[3])
    for sl in (slice(0, 1), slice(1, 4), slice(4, 31)):
        scale = np.max(np.abs(b[1][:, sl]), axis=1, keepdims=True)
        assert np.all(np.abs(a[1][:, sl] - b[1][:, sl]) <= 1e-3 * scale)
