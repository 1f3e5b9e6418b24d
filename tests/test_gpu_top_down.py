"""Grid and k-section searches that stop the candidates below one that passed
(early exit per candidate) against the same searches with early exit per
trajectory, which run every candidate: equal results over scenario counts around
a block, a warp and a wave, every kernel form, and recheck bands wide enough that
passing candidates are undecided."""
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


TARGETS = [(100.0, 250.0, 1.0), (200.0, 60.0, 1.0), (100.0, 180.0, 1.002), (150.0, 152.0, 0.995)]


@pytest.mark.parametrize("N", [1, 33, 128, 5000, 20001])
@pytest.mark.parametrize("search", ["SEARCH_GRID", "SEARCH_KSECTION"])
@pytest.mark.parametrize("form", ["fp64", "fp32", "recheck", "wide_band", "in_register", "tma", "pairs", "uncertain"])
def test_result_equals_running_every_candidate(R, orc, params, N, search, form):
    if form == "tma":
        N = (N + 3) // 4 * 4
    if form == "fp64" and N > 128:
        N = 300
    kw = dict(horizon=150, n_scenarios=N, max_candidates=16, n_rounds=3, search=getattr(R, search),
              precision={"fp64": R.FP64, "fp32": R.FP32}.get(form, R.FP32_RECHECK),
              scenarios_in_register=int(form == "in_register"), param_unc_rel=0.1 if form == "uncertain" else 0.0,
              recheck_eps_rel=1e-2 if form == "wide_band" else 1e-5)
    got = []
    for early in (R.EXIT_LANE, R.EXIT_CANDIDATE):
        with R.Governor(params, R.rrg_config_default(early_exit=early, **kw)) as g:
            if form == "tma":
                g.set_tma(2)
            if form == "pairs":
                g.set_pairing(2)
            for t, (v, r, f) in enumerate(TARGETS):
                g.sample_scenarios(3, t)
                got.append(g.step(orc.equilibrium(params, v) * f, r, v))
    assert got[:len(TARGETS)] == got[len(TARGETS):]


@pytest.mark.parametrize("S,M", [(1, 2), (7, 16), (40, 32)])
@pytest.mark.parametrize("search", ["SEARCH_GRID", "SEARCH_KSECTION"])
@pytest.mark.parametrize("band", [1e-5, 1e-2])
def test_batch_equals_running_every_candidate(R, orc, params, S, M, search, band):
    rng = np.random.default_rng(S)
    N, H = rng.integers(1, 700, S), rng.integers(1, 200, S)
    v = rng.uniform(60.0, 250.0, S)
    r = rng.uniform(60.0, 280.0, S)
    x = np.array([orc.equilibrium(params, a) for a in v])
    out = []
    for early in (R.EXIT_LANE, R.EXIT_CANDIDATE):
        cfg = R.rrg_config_default(max_candidates=M, n_rounds=3, search=getattr(R, search), early_exit=early,
                                   precision=R.FP32_RECHECK, recheck_eps_rel=band)
        with R.BatchGovernor(params, cfg, N, H) as g:
            for var in range(10):
                g.set_variant(var)
                out.append(g.step(x, r, v, 5, 1))
    for o in out[1:]:
        for a, b in zip(out[0], o):
            np.testing.assert_array_equal(a, b)
