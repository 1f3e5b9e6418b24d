"""The power tables that the allocation-free evaluation keeps in its scratch: results
over more exponents than it keeps, in any order, and in a captured call whose exponent
was not met before, equal a handle's; models in turn cost no more than one."""
import time

import numpy as np
import pytest

from paper_2510_08288_gb300 import inputs

pytestmark = pytest.mark.gpu

N, H, M = 40, 60, 4
KAPPAS = np.linspace(0.0, 0.6, M)


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_08288_gb300 import build as B
    B.build()
    from paper_2510_08288_gb300 import rrg
    return rrg


class Static:
    def __init__(self, R, precision):
        import torch
        self.R, self.torch = R, torch
        self.cfg = R.rrg_config_default(horizon=H, n_scenarios=N, max_candidates=M, precision=precision,
                                        early_exit=R.EXIT_NONE, recheck_eps_rel=1e-1)
        self.d = inputs.uniform_disturbances(N, H, 5)
        self.d64 = torch.tensor(self.d, device="cuda")
        self.d32 = self.d64.float()
        self.k = torch.tensor(KAPPAS, device="cuda")
        self.adm = torch.zeros(M, dtype=torch.uint8, device="cuda")
        self.ms = torch.zeros(M, dtype=torch.float64, device="cuda")
        self.x = torch.zeros(3, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()

    def call(self, p, stream):
        self.R.rrg_eval_candidates_static(p, self.cfg, stream, self.d64, self.d32, self.x, 100.0, 250.0, self.k, M,
                                          self.adm, self.ms)

    def handle(self, p):
        with self.R.Governor(p, self.cfg) as g:
            g.set_scenarios(self.d)
            x, _ = g.equilibrium(100.0)
            a, s, _ = g.eval_candidates(x, 100.0, 250.0, KAPPAS)
        return x, a, s

    def check(self, p, run):
        x, a, s = self.handle(p)
        self.x.copy_(self.torch.tensor(x))
        self.torch.cuda.synchronize()
        run()
        self.torch.cuda.synchronize()
        np.testing.assert_array_equal(self.adm.cpu().numpy(), a)
        np.testing.assert_array_equal(self.ms.cpu().numpy(), s)


@pytest.mark.parametrize("precision", [0, 2])
def test_more_exponents_than_are_kept(R, precision):
    """Binary64, and binary32 with nearly every trajectory rechecked in binary64."""
    S = Static(R, precision)
    stream = S.torch.cuda.Stream()
    gammas = [1.4 - 0.004 * i for i in range(12)]
    for g in gammas + gammas[::-1] + [1.4, 1.36, 1.4]:
        p = inputs.fc3_params(gamma=g)
        S.check(p, lambda: S.call(p, stream))


def test_captured_call_with_an_exponent_first_met_in_the_capture(R):
    S = Static(R, R.FP64)
    stream = S.torch.cuda.Stream()
    S.call(inputs.fc3_params(), stream)  # (the first call, before any capture)
    stream.synchronize()
    models = [inputs.fc3_params(gamma=g) for g in (1.4, 1.3123)]
    graphs = []
    for p in models:
        graph = S.torch.cuda.CUDAGraph()
        with S.torch.cuda.graph(graph, stream=stream):
            S.call(p, stream)
        graphs.append(graph)
    other = inputs.fc3_params(gamma=1.2987)
    for _ in range(2):
        for p, graph in zip(models, graphs):
            S.check(p, graph.replay)
        S.check(other, lambda: S.call(other, stream))
        S.check(models[1], lambda: S.call(models[1], stream))


def test_models_in_turn_cost_no_more_than_one(R):
    S = Static(R, R.FP32_RECHECK)
    stream = S.torch.cuda.Stream()
    p, q = inputs.fc3_params(), inputs.fc3_params(gamma=1.4 - 0.004)

    def host_us(models):
        t = []
        for i in range(220):
            stream.synchronize()
            t0 = time.perf_counter()
            S.call(models[i & 1], stream)
            t.append(time.perf_counter() - t0)
        return np.median(t[20:]) * 1e6
    one, turn = host_us((p, p)), host_us((p, q))
    print("host time of a call: one model %.1f us, two in turn %.1f us" % (one, turn))
    assert turn < 1.25 * one
