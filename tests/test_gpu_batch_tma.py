"""The batched rollouts on the per-warp TMA ring, forced, against the register
forms: scenario counts that are no multiple of 4 or 32, horizons around the
16-step chunk, every early exit, both scenario pairs of the closed loop, and
searches whose rows run from the largest candidate down."""
import numpy as np
import pytest

from paper_2510_08288_gb300 import inputs

pytestmark = pytest.mark.gpu

N = [1, 2, 3, 5, 31, 32, 33, 63, 127, 129, 130, 258]
H = [1, 15, 16, 17, 31, 33, 48, 2, 100, 16, 7, 64]
RING = (1, 3, 5, 7)  # the variants of prefetch depth 16


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_08288_gb300 import build as B
    B.build()
    from paper_2510_08288_gb300 import rrg
    return rrg


def _problems(orc, params, S):
    rng = np.random.default_rng(4)
    vp, r = rng.uniform(80, 180, S), rng.uniform(90, 300, S)
    x = np.array([orc.equilibrium(params, v) for v in vp]) + rng.uniform(-150, 150, (S, 3)) * [1, 0.1, 1]
    return x, r, vp


def _config(R, search, **kw):
    more = dict(search=R.SEARCH_KSECTION, n_rounds=2) if search == "ksection" else dict(search=R.SEARCH_SPEC_BISECT)
    return R.rrg_config_default(max_candidates=8, precision=R.FP32_RECHECK, **more, **kw)


@pytest.mark.parametrize("early_exit", [0, 1, 2])
@pytest.mark.parametrize("search", ["ksection", "spec"])
def test_tma_ring_equals_register_form(R, orc, params, early_exit, search):
    S, T = len(N), 3
    x, r, vp = _problems(orc, params, S)
    amp = np.array(inputs.DIST_AMP)
    with R.BatchGovernor(params, _config(R, search, early_exit=early_exit), N, H) as g:
        assert g.get_tma() == R.TMA_AUTO

        def run():
            return (*g.step(x, r, vp, 21, 5), *g.closed_loop(x, vp, np.tile(r, (T, 1)), 21, 5, amp))
        g.set_variant(0)
        want = run()
        for mode in (R.TMA_ALWAYS, R.TMA_NEVER):
            g.set_tma(mode)
            assert g.get_tma() == mode
            for var in RING:
                g.set_variant(var)
                g.reset_stats()
                got = run()
                st = g.stats()
                assert st["lane_steps_tma"] + st["lane_steps_fp64"] == (st["lane_steps"] if mode else
                                                                        st["lane_steps_fp64"])
                assert (st["lane_steps_tma"] > 0) == (mode == R.TMA_ALWAYS) and st["wait_timeouts"] == 0
                for a, b in zip(want, got):
                    np.testing.assert_array_equal(a, b)
        for bad in (-1, 3):
            with pytest.raises(R.RrgError):
                g.set_tma(bad)


def test_rounds_of_many_tiles_take_the_tma_ring(R, orc, params):
    """RRG_TMA_AUTO: 1,024 candidates of 1,000 warps of scenarios reach 300
    warps of tiles per SM, 8 candidates of the same do not; equal results."""
    x, r, vp = _problems(orc, params, 1)
    out = []
    for M in (8, 1024):
        cfg = R.rrg_config_default(max_candidates=M, precision=R.FP32_RECHECK, search=R.SEARCH_GRID,
                                   early_exit=R.EXIT_CANDIDATE)
        with R.BatchGovernor(params, cfg, [32000], [20]) as g:
            g.step(x, r, vp, 21, 5)
            assert (g.stats()["lane_steps_tma"] > 0) == (M == 1024)
            a = g.step(x, r, vp, 21, 5)
            g.set_tma(R.TMA_NEVER if M == 1024 else R.TMA_ALWAYS)
            out.append((a, g.step(x, r, vp, 21, 5)))
    for a, b in out:
        for u, w in zip(a, b):
            np.testing.assert_array_equal(u, w)


@pytest.mark.parametrize("variant", RING)
def test_a_warp_that_gave_up_leaves_the_ring(R, orc, params, variant):
    """Without copies (RRG_INJECT_TMA_NO_COPY) each warp's wait runs out once: its
    tile and the many that it takes afterwards count as violated, none of them on
    the ring again.  Nothing is admissible, and the handle recovers."""
    import torch
    warps = 64 * torch.cuda.get_device_properties(0).multi_processor_count
    cfg = R.rrg_config_default(max_candidates=16, precision=R.FP32_RECHECK, search=R.SEARCH_GRID,
                               early_exit=R.EXIT_LANE)
    x, r, vp = _problems(orc, params, 1)
    with R.BatchGovernor(params, cfg, [64000], [48]) as g:
        g.set_variant(variant)
        g.set_tma(R.TMA_ALWAYS)
        want = g.step(x, r, vp, 21, 5)
        g.set_injection(R.INJECT_TMA_NO_COPY)
        g.reset_stats()
        _, kappa, flags = g.step(x, r, vp, 21, 5)
        st = g.stats()
        assert 0 < st["wait_timeouts"] <= warps < 16 * 2000  # once a warp; 2,000 warps of tiles a candidate
        assert kappa[0] == 0.0 and flags[0] & 1 and want[1][0] > 0.0
        assert st["lane_steps"] == 0
        g.set_injection(0)
        g.reset_stats()
        for a, b in zip(want, g.step(x, r, vp, 21, 5)):
            np.testing.assert_array_equal(a, b)
        assert g.stats()["wait_timeouts"] == 0
        with pytest.raises(R.RrgError):
            g.set_injection(2)
