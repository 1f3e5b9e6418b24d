"""The batched rollouts on the per-warp TMA ring (variants of prefetch depth
16) against the register forms, at scenario counts that are no multiple of 4 or
32 and horizons around the 16-step chunk."""
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


N = [1, 2, 3, 5, 31, 32, 33, 63, 127, 129, 130, 258]
H = [1, 15, 16, 17, 31, 33, 48, 2, 100, 16, 7, 64]


@pytest.mark.parametrize("early_exit", [0, 1, 2])
@pytest.mark.parametrize("search", ["ksection", "spec"])
def test_ring_variants_equal_register_variants_and_oracle(R, orc, params, early_exit, search):
    S = len(N)
    rng = np.random.default_rng(4)
    vp, r = rng.uniform(80, 180, S), rng.uniform(90, 300, S)
    x = np.array([orc.equilibrium(params, v) for v in vp]) + rng.uniform(-150, 150, (S, 3)) * [1, 0.1, 1]
    kw = dict(search=R.SEARCH_KSECTION, n_rounds=2) if search == "ksection" else dict(search=R.SEARCH_SPEC_BISECT)
    cfg = R.rrg_config_default(max_candidates=8, precision=R.FP32_RECHECK, early_exit=early_exit, **kw)
    T = 3
    amp = np.array(inputs.DIST_AMP)
    with R.BatchGovernor(params, cfg, N, H) as g:
        out = []
        for var in (0, 1, 3, 5, 7):
            g.set_variant(var)
            one = g.step(x, r, vp, 21, 5)
            loop = g.closed_loop(x, vp, np.tile(r, (T, 1)), 21, 5, amp)  # both scenario pairs
            out.append((*one, *loop))
        assert g.stats()["wait_timeouts"] == 0
    for o in out[1:]:
        for a, b in zip(out[0], o):
            np.testing.assert_array_equal(a, b)
    for s in range(S):
        d = orc.sample_disturbances(21 + s, 5, N[s], H[s], inputs.DIST_AMP)
        c = orc.cfg(H=H[s], N=N[s])
        if search == "ksection":
            k, f = orc.ksection(params, c, x[s], vp[s], r[s], 8, 2, d)
        else:
            k, f = orc.bisect_joint(params, c, x[s], vp[s], r[s], 12, d)
        assert out[0][1][s] == k and out[0][2][s] == f
