"""A call that fails after its first kernels are queued returns only once they have
run: they read and write the handle's pinned staging, which the next call writes."""
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


CALLS = {
    "eval": lambda g, x: g.eval_candidates(x, 100.0, 150.0, [0.0, 0.5, 1.0]),
    "gradient": lambda g, x: g.slack_gradients(x, 100.0, 150.0, [0.1, 0.4]),
    "newton": lambda g, x: g.newton_search(x, 150.0, 100.0, 1e-3),
    "step": lambda g, x: g.step(x, 150.0, 100.0),
}


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("profiling", [False, True])
def test_error_return_leaves_nothing_queued(R, orc, params, call, profiling):
    import torch
    x = orc.equilibrium(params, 100.0)
    stream = torch.cuda.Stream()
    with R.Governor(params, R.rrg_config_default(horizon=60, n_scenarios=64, max_candidates=16), stream) as g:
        g.sample_scenarios(1, 0)
        want = CALLS[call](g, x)
        g.set_profiling(profiling)  # (direct launches instead of a graph)
        g.set_injection(R.INJECT_LAUNCH_ERROR)
        stream.synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(1 << 28)
        with pytest.raises(R.RrgError) as e:
            CALLS[call](g, x)
        assert e.value.code == R.RRG_ECUDA
        assert stream.query()
        g.set_injection(0)
        for a, b in zip(want, CALLS[call](g, x)):
            np.testing.assert_array_equal(a, b)
