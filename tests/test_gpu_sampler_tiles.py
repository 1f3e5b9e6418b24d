"""The tiled scenario sampler (steps x scenarios per block, the parts of a
Philox block that depend on one of them formed once) at the remainders of its
tiles, against the oracle's draws and against lanes that draw block by block."""
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


SHAPES = [(1, 1), (1, 70000), (31, 65), (32, 3), (33, 129), (64, 64), (65, 7), (255, 130), (257, 33), (300, 1)]


@pytest.mark.parametrize("N,H", SHAPES)
@pytest.mark.parametrize("seed,update,base", [(7, 0, 0), (2**64 - 3, 2**40 + 1, 2**33 + 5)])
def test_draws_equal_the_oracle(R, orc, params, N, H, seed, update, base):
    """Both binary64 forms, drawn (RRG_FP64) and regenerated (a binary32
    handle), equal a (2u - 1) of the counters (j, base + k, update, 0) bit for
    bit; a row of the counters is recomputed by numpy's Philox."""
    got = []
    for prec in (R.FP64, R.FP32_RECHECK):
        cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=2, precision=prec, scenario_base=base)
        with R.Governor(params, cfg) as g:
            g.sample_scenarios(seed, update)
            got.append(g.get_scenarios())
    np.testing.assert_array_equal(got[0], got[1])
    if base == 0:
        np.testing.assert_array_equal(got[0], orc.sample_disturbances(seed, update, N, H, inputs.DIST_AMP))
    k = N - 1
    c = ((base + k) << 64 | update << 128) - 1
    words = np.array([(c >> (64 * i)) & (2**64 - 1) for i in range(4)], dtype=np.uint64)
    raw = np.random.Philox(key=np.array([seed, 0], dtype=np.uint64), counter=words).random_raw(4 * H)
    u = (raw.reshape(H, 4)[:, :3] >> np.uint64(11)) * 2.0**-53
    np.testing.assert_array_equal(got[0][:, :, k].T, np.array(inputs.DIST_AMP) * (2.0 * u - 1.0))


@pytest.mark.parametrize("N,H", [s for s in SHAPES if s[1] < 1000])
def test_binary32_copy_equals_the_draw_in_the_loop(R, params, N, H):
    """Trajectories on the stored binary32 copy equal those whose lanes draw
    each block in the trajectory loop."""
    kap = np.array([0.0, 0.05, 0.3])
    out = []
    for gen in (0, 1):
        cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=4, precision=R.FP32, early_exit=0,
                                   scenarios_in_register=gen)
        with R.Governor(params, cfg) as g:
            x, _ = g.equilibrium(100.0)
            g.sample_scenarios(5, 9)
            out.append(g.eval_candidates(x, 100.0, 160.0, kap, want_P=True))
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
