"""Grid and k-section updates whose candidates violate late, whose launches come in
two parts (held to one candidate's warps, then at full residency): results equal
running every candidate, and an update without an admissible candidate takes no
much longer than evaluating its candidates all at once."""
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


def _cfg(R, N, y_min, **kw):
    base = dict(horizon=4000, n_scenarios=N, max_candidates=16, n_rounds=3, search=R.SEARCH_KSECTION,
                precision=R.FP32_RECHECK, ss_check=0, y_min=y_min, param_unc_rel=0.1)
    base.update(kw)
    return R.rrg_config_default(**base)


@pytest.mark.parametrize("N", [7264, 7296, 16384, 16385, 27232, 32768, 35000])
@pytest.mark.parametrize("y_min", [1.92, 1.94, 1.95])
@pytest.mark.parametrize("form", ["recheck", "fp32", "tma", "nominal", "grid"])
def test_result_equals_running_every_candidate(R, params, N, y_min, form):
    kw = dict(horizon=1000)
    if form == "fp32":
        kw.update(precision=R.FP32)
    if form == "nominal":
        kw.update(param_unc_rel=0.0)
        y_min += 0.22  # (nominal scenarios stay closer to the setpoint's output)
    if form == "grid":
        kw.update(search=R.SEARCH_GRID)
    out = []
    for early in (R.EXIT_LANE, R.EXIT_CANDIDATE):
        with R.Governor(params, _cfg(R, N, y_min, early_exit=early, **kw)) as g:
            if form == "tma" and N % 4 == 0:
                g.set_tma(R.TMA_ALWAYS)
            x, _ = g.equilibrium(200.0)
            for t in range(2):
                g.sample_scenarios(1, t)
                out.append(g.step(x, 100.0, 200.0))
    assert out[:2] == out[2:]


@pytest.mark.parametrize("N", [13000, 16384])
def test_update_without_admissible_candidate_is_not_slower(R, params, N):
    with R.Governor(params, _cfg(R, N, 1.945)) as g:
        x, _ = g.equilibrium(200.0)
        g.set_profiling(True)
        ms = {"step": [], "every candidate": []}
        for t in range(9):
            g.sample_scenarios(1, 1)
            g.reset_stats()
            if t % 2:
                _, kappa, flags = g.step(x, 100.0, 200.0)
                assert kappa == 0.0 and flags & 1
            else:
                adm, _, _ = g.eval_candidates(x, 200.0, 100.0, np.linspace(0.0, 1.0, 16))
                assert not adm.any()
            ms["step" if t % 2 else "every candidate"].append(g.stats()["rollout_ms"])
    print({k: np.median(v) for k, v in ms.items()})
    assert np.median(ms["step"]) < 1.7 * np.median(ms["every candidate"][1:])
