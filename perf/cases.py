"""What a user of the robust reference governor has it do, as measurable cases.

Every case is one call (or the draw-and-search pair that makes one governor
update) through the public Python binding: a control tick, a simulated closed
loop, an evaluation of given candidates, a gradient of the robust objective, an
update of many governors at once, a Monte Carlo sweep.  Sizes are those of the
workloads in paper_2510_08288_gb300/inputs.py and of the tests, with odd and
ragged ones beside them.

Inputs: the setpoints lie in the 50..300 A range that the model is meant for,
and the measured state is the equilibrium of the last setpoint moved by as much
as the disturbances move it (batched instances: by up to 10 % per component, as
inputs.batched_instances draws them).

Numbers that the framework computes in binary32 (the min slacks and gradients of
its binary32 modes, which the C ABI carries in doubles) are returned as binary32;
setpoints, kappas and plant states are binary64 and are returned as that.

exact() restates the model (FC3, RK4, the Philox draws) in plain numpy and torch
in binary64.
"""
import math

import numpy as np
import torch

from paper_2510_08288_gb300 import inputs
from paper_2510_08288_gb300 import rrg as R

SEARCH = {"bisect": R.SEARCH_BISECT, "ksection": R.SEARCH_KSECTION, "spec": R.SEARCH_SPEC_BISECT}
PRECISION = {"fp64": R.FP64, "fp32+recheck": R.FP32_RECHECK}


def listed():
    return [
        # the governor inside a 10 ms control task: 32 scenarios, 500 steps, the library's defaults
        {"name": "tick_n32", "kind": "update", "N": 32, "H": 500, "M": 32, "search": "spec",
         "precision": "fp32+recheck", "unc": 0.0, "in_register": False},
        # the same update as the paper writes it: serial bisection, everything in binary64
        {"name": "tick_fp64_n32", "kind": "update", "N": 32, "H": 500, "M": 1, "search": "bisect",
         "precision": "fp64", "unc": 0.0, "in_register": False},
        # an update that stores no scenario array (device memory kept for other work)
        {"name": "update_in_register_n1000", "kind": "update", "N": 1000, "H": 2000, "M": 64, "search": "spec",
         "precision": "fp32+recheck", "unc": 0.0, "in_register": True},
        # a governed run against the simulated plant: 1,024 scenarios, 2,000 steps, reference levels up and down
        {"name": "loop_n1024", "kind": "loop", "N": 1024, "H": 2000, "M": 64, "T": 16, "hold": 4},
        # the admissibility matrix P and the min slacks of a whole kappa grid, an odd scenario count
        {"name": "eval_n3001", "kind": "eval", "N": 3001, "H": 1000, "M": 32, "precision": "fp32+recheck", "unc": 0.0},
        # the same in binary64, as the reference that a binary32 result is checked with
        {"name": "eval_fp64_n257", "kind": "eval", "N": 257, "H": 500, "M": 8, "precision": "fp64", "unc": 0.0},
        # one gradient of the robust objective (a step of a design or tuning loop)
        {"name": "gradient_fp32_n4096", "kind": "gradient", "N": 4096, "H": 1000, "m": 1, "checkpoint": 50,
         "precision": "fp32"},
        # gradients at several kappas in binary64
        {"name": "gradient_fp64_n1024", "kind": "gradient", "N": 1024, "H": 1000, "m": 3, "checkpoint": 50,
         "precision": "fp64"},
        # one update of 64 independent governors of very different sizes
        {"name": "batch_s64", "kind": "batch", "S": 64, "N_lo": 64, "N_hi": 8192, "H_lo": 200, "H_hi": 4000, "M": 32,
         "search": "ksection"},
        # closed loops of 16 governors, bisection result, small trees
        {"name": "batch_loop_s16", "kind": "batch_loop", "S": 16, "N_lo": 64, "N_hi": 2048, "H_lo": 200,
         "H_hi": 2000, "M": 7, "search": "spec", "T": 4},
        # Monte Carlo robustness sweep, disturbances and uncertain parameters, 5,000 steps: middle and largest
        {"name": "sweep_n16384", "kind": "update", "N": 16384, "H": 5000, "M": 16, "search": "ksection",
         "precision": "fp32+recheck", "unc": 0.1, "in_register": False},
        {"name": "sweep_n65536", "kind": "update", "N": 65536, "H": 5000, "M": 16, "search": "ksection",
         "precision": "fp32+recheck", "unc": 0.1, "in_register": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("tick", "update", "sweep", "loop", "eval", "eval_fp64", "gradient", "gradient_fp64", "batch",
                       "batch_loop"))
    if kind == "tick":
        fp64 = rng.random() < 0.3
        return {"kind": "update", "N": _log(rng, 1, 512 if not fp64 else 64),
                "H": rng.randint(100, 400 if fp64 else 1000), "M": 1 if fp64 else rng.choice((7, 16, 32, 64)), "search": "bisect" if fp64 else "spec",
                "precision": "fp64" if fp64 else "fp32+recheck", "unc": 0.0, "in_register": False}
    if kind == "update":
        return {"kind": "update", "N": _log(rng, 200, 8192), "H": rng.randint(500, 4000),
                "M": rng.choice((16, 32, 64)), "search": rng.choice(("spec", "ksection")),
                "precision": "fp32+recheck", "unc": rng.choice((0.0, 0.05)), "in_register": rng.random() < 0.3}
    if kind == "sweep":
        n = _log(rng, 1000, 40000)
        return {"kind": "update", "N": n if rng.random() < 0.4 else (n + 63) // 64 * 64, "H": rng.randint(2000, 5000),
                "M": 16, "search": "ksection", "precision": "fp32+recheck", "unc": rng.choice((0.0, 0.1)),
                "in_register": False}
    if kind == "loop":
        return {"kind": "loop", "N": _log(rng, 30, 2048), "H": rng.randint(300, 2500),
                "M": rng.choice((16, 32, 64)), "T": rng.randint(4, 16), "hold": rng.randint(2, 5)}
    if kind == "eval":
        return {"kind": "eval", "N": _log(rng, 33, 8192), "H": rng.randint(200, 1500), "M": rng.randint(1, 32),
                "precision": "fp32+recheck", "unc": rng.choice((0.0, 0.1))}
    if kind == "eval_fp64":
        return {"kind": "eval", "N": _log(rng, 17, 600), "H": rng.randint(100, 700), "M": rng.randint(1, 8),
                "precision": "fp64", "unc": rng.choice((0.0, 0.1))}
    if kind == "gradient":
        return {"kind": "gradient", "N": _log(rng, 100, 8192), "H": rng.randint(200, 1500), "m": rng.randint(1, 4),
                "checkpoint": rng.choice((16, 50, 100)), "precision": "fp32"}
    if kind == "gradient_fp64":
        return {"kind": "gradient", "N": _log(rng, 64, 2048), "H": rng.randint(100, 900), "m": rng.randint(1, 3),
                "checkpoint": rng.choice((16, 50, 100)), "precision": "fp64"}
    if kind == "batch":
        return {"kind": "batch", "S": rng.randint(2, 48), "N_lo": 64, "N_hi": rng.randint(500, 8192), "H_lo": 200,
                "H_hi": rng.randint(500, 4000), "M": rng.choice((8, 16, 32)),
                "search": rng.choice(("ksection", "spec"))}
    return {"kind": "batch_loop", "S": rng.randint(2, 24), "N_lo": 32, "N_hi": rng.randint(200, 2048), "H_lo": 100,
            "H_hi": rng.randint(300, 2000), "M": rng.choice((3, 7, 15)), "search": "spec", "T": rng.randint(2, 5)}


def _config(case):
    unc = case.get("unc", 0.0)
    kw = dict(horizon=case["H"], n_scenarios=case["N"], precision=PRECISION.get(case.get("precision"), R.FP32_RECHECK),
              param_unc_rel=unc, param_unc_mask=inputs.FC3_UNCERTAIN_MASK, recheck_eps_rel=1e-6)
    if case["kind"] == "gradient":
        kw.update(max_candidates=max(4, case["m"]),
                  precision=R.FP64 if case["precision"] == "fp64" else R.FP32_RECHECK)
    elif case["kind"] == "eval":
        # every trajectory over the whole horizon: the min slacks are then the minima themselves
        kw.update(max_candidates=case["M"], early_exit=R.EXIT_NONE)
    else:
        kw.update(max_candidates=case["M"], search=SEARCH[case.get("search", "spec")],
                  scenarios_in_register=int(case.get("in_register", False)))
    return R.rrg_config_default(**kw)


def _measured_state(g, v_prev, rng):
    """The equilibrium of the last setpoint, as far from it as a few disturbances take it."""
    x, _ = g.equilibrium(v_prev)
    return x + np.array([150.0, 20.0, 150.0]) * rng.uniform(-1.0, 1.0, 3)


def _batch_inputs(case, rng):
    b = inputs.batched_instances(case["S"], int(rng.integers(1 << 31)), case["N_lo"], case["N_hi"], case["H_lo"],
                                 case["H_hi"])
    with R.Governor(inputs.fc3_params(), R.rrg_config_default(horizon=1, n_scenarios=1)) as g:
        x_eq = np.array([g.equilibrium(v)[0] for v in b["v_prev"]])
    return b, x_eq * b["xfac"]


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    p = inputs.fc3_params()
    s = {"case": case, "seed": int(rng.integers(1 << 40)), "update": int(rng.integers(1 << 20))}
    kind = case["kind"]
    if kind in ("batch", "batch_loop"):
        b, s["x"] = _batch_inputs(case, rng)
        cfg = R.rrg_config_default(max_candidates=case["M"], search=SEARCH[case["search"]], n_rounds=3,
                                   precision=R.FP32_RECHECK, recheck_eps_rel=1e-6)
        s["g"] = R.BatchGovernor(p, cfg, b["N"], b["H"])
        s["v_prev"], s["r"] = b["v_prev"], b["r"]
        if kind == "batch_loop":
            s["r"] = np.tile(b["r"], (case["T"], 1))
        return s
    s["g"] = g = R.Governor(p, _config(case))
    s["v_prev"] = v_prev = float(rng.uniform(80.0, 180.0))
    s["x"] = _measured_state(g, v_prev, rng)
    if kind == "loop":
        T = case["T"]
        s["r"] = inputs.staircase(T, -(-T // case["hold"]), case["hold"], int(rng.integers(1 << 31)))
        return s
    s["r"] = v_prev + float(rng.uniform(20.0, 120.0))  # the load rises: the direction that the constraint limits
    if kind == "eval":
        s["kappas"] = np.sort(rng.uniform(0.0, 1.0, case["M"])) ** 2
    if kind == "gradient":
        s["kappas"] = np.sort(rng.uniform(0.02, 0.9, case["m"]))
    if kind in ("eval", "gradient"):
        g.sample_scenarios(s["seed"], s["update"])
    return s


def run(s):
    case, g = s["case"], s["g"]
    kind = case["kind"]
    if kind == "update":
        g.sample_scenarios(s["seed"], s["update"])
        v, kappa, flags = g.step(s["x"], s["r"], s["v_prev"])
        return {"v": v, "kappa": kappa, "flags": flags}
    if kind == "loop":
        v, kappa, flags, x = g.closed_loop(s["x"], s["v_prev"], s["r"], s["seed"], s["update"], inputs.DIST_AMP)
        return {"v": v, "kappa": kappa, "flags": flags, "x": x}
    if kind == "eval":
        adm, slack, P = g.eval_candidates(s["x"], s["v_prev"], s["r"], s["kappas"], want_P=True)
        return {"admissible": adm, "min_slack": slack if case["precision"] == "fp64" else slack.astype(np.float32),
                "P": P}
    if kind == "gradient":
        fp64 = case["precision"] == "fp64"
        val, grad, k, j, ss = g.slack_gradients(s["x"], s["v_prev"], s["r"], s["kappas"], case["checkpoint"],
                                                R.FP64 if fp64 else R.FP32)
        if not fp64:
            val, grad = val.astype(np.float32), grad.astype(np.float32)
        return {"g": val, "grad": grad, "k": k, "j": j, "ss_ok": ss}
    if kind == "batch":
        v, kappa, flags = g.step(s["x"], s["r"], s["v_prev"], s["seed"], s["update"])
        return {"v": v, "kappa": kappa, "flags": flags}
    v, kappa, flags, x = g.closed_loop(s["x"], s["v_prev"], s["r"], s["seed"], s["update"], inputs.DIST_AMP)
    return {"v": v, "kappa": kappa, "flags": flags, "x": x}


# One RK4 step of a trajectory: 4 right-hand sides of 24 operations, 3 stage points of 6, the combination 18, the
# disturbance 3, output, slack and running minimum 6.
STEP_FLOPS = 141.0
# One step's sample of a scenario's disturbances: 10 Philox rounds of two 64 x 64 -> 128 bit products, as operations.
DRAW_FLOPS = 40.0


def work(case):
    """The trajectories that the result cannot do without: every one of them where all values are returned, those of
    the chosen candidate in a search; a draw of the scenarios where the call makes one.  Bytes: what the call returns,
    and the scenarios where the caller holds them already."""
    kind = case["kind"]
    if kind in ("batch", "batch_loop"):
        # the expected sum of N_s H_s over the instances (log-uniform N, uniform H)
        lo, hi = case["N_lo"], case["N_hi"]
        n = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        steps = case["S"] * n * 0.5 * (case["H_lo"] + case["H_hi"]) * case.get("T", 1)
        return {"bytes": 44.0 * case["S"] * case.get("T", 1), "flops": steps * (STEP_FLOPS + DRAW_FLOPS)}
    steps = float(case["N"]) * case["H"]
    if kind == "eval":
        return {"bytes": 12.0 * steps + case["M"] * (case["N"] + 9.0), "flops": case["M"] * steps * STEP_FLOPS}
    if kind == "gradient":
        return {"bytes": 12.0 * steps + case["m"] * 35 * 8.0, "flops": case["m"] * steps * STEP_FLOPS}
    T = case.get("T", 1)
    return {"bytes": 44.0 * T, "flops": T * steps * (STEP_FLOPS + DRAW_FLOPS)}


# ---------------------------------------------------------------- 64-bit restatement of the model
_NAMES = {n: i for i, n in enumerate(inputs.FC3_PARAM_NAMES)}


def _consts(P, v):
    """Flow of oxygen consumed, motor voltage at zero flow error and OER per pascal at setpoint v."""
    w_o2 = P["M_O2"] * P["n_cell"] * v / (4.0 * P["faraday"])
    v0 = P["c0"] + P["c1"] * v + P["c2"] * v * v + P["K_p"] * P["lam_ref"] * w_o2 / P["x_O2"]
    return w_o2, v0, P["x_O2"] * P["k_sm"] / w_o2


def _rhs(P, c, ca, w, sm):
    w_o2, v0, _ = c
    w_cp = P["a_w"] * w - P["a_p"] * sm
    w_sm = P["k_sm"] * (sm - ca)
    pr = (1.0 + sm / P["p_atm"]) ** ((P["gamma"] - 1.0) / P["gamma"]) - 1.0
    t_cp = P["c_p"] * P["T_atm"] / P["eta_cp"] * pr * w_cp / w
    t_cm = P["eta_cm"] * P["k_t"] / P["R_cm"] * (v0 - P["K_p"] * w_cp - P["k_v"] * w)
    rt = P["R_a"] * P["T_st"]
    return rt / P["V_ca"] * (w_sm - P["k_ca"] * ca - w_o2), (t_cm - t_cp) / P["J_cp"], rt / P["V_sm"] * (w_cp - w_sm)


def _rk4(P, c, q, dt=inputs.DT):
    def at(k, h):
        return [a + h * b for a, b in zip(q, k)]
    k1 = _rhs(P, c, *q)
    k2 = _rhs(P, c, *at(k1, 0.5 * dt))
    k3 = _rhs(P, c, *at(k2, 0.5 * dt))
    k4 = _rhs(P, c, *at(k3, dt))
    return [a + dt / 6.0 * (b1 + 2.0 * (b2 + b3) + b4) for a, b1, b2, b3, b4 in zip(q, k1, k2, k3, k4)]


def _philox(seed, stream, k, update, blocks):
    """Words [blocks, 4] of Philox4x64-10 at counters (0.., k, update, stream); numpy adds one before each block."""
    c = ((k << 64) | (update << 128) | (stream << 192)) - 1
    words = np.array([(c >> (64 * i)) & (2 ** 64 - 1) for i in range(4)], dtype=np.uint64)
    bg = np.random.Philox(key=np.array([seed, 0], dtype=np.uint64), counter=words)
    return bg.random_raw(4 * blocks).reshape(blocks, 4)


def _sym(words):
    return 2.0 * ((words >> np.uint64(11)) * 2.0 ** -53) - 1.0


def _disturbances(seed, update, N, H):
    d = np.empty((3, H, N))
    for k in range(N):
        d[:, :, k] = _sym(_philox(seed, 0, k, update, H))[:, :3].T
    return d * np.array(inputs.DIST_AMP).reshape(3, 1, 1)


def _model(seed, update, N, rho, dev):
    """Parameters by name, each a number, or a row over the scenarios where it is uncertain."""
    P = dict(inputs.FC3_DEFAULTS)
    if rho:
        groups = -(-len(_NAMES) // 4)
        u = np.stack([_sym(_philox(seed, 2, k, update, groups)).reshape(-1) for k in range(N)])
        for n in inputs.FC3_UNCERTAIN:
            P[n] = torch.as_tensor(P[n] * (1.0 + rho * u[:, _NAMES[n]]), device=dev).reshape(1, N)
    return P


def _steady_ok(v, y_min=inputs.Y_MIN, eps=0.05, y_c=2.2):
    """Eq. 3's check of one setpoint at the nominal model: the equilibrium by bisection on the air flow."""
    P = inputs.FC3_DEFAULTS
    c = _consts(P, v)

    def state(W):
        ca = (W - c[0]) / P["k_ca"]
        sm = ca + W / P["k_sm"]
        return ca, (W + P["a_p"] * sm) / P["a_w"], sm

    lo, hi = c[0], 20.0 * c[0] / P["x_O2"]
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if _rhs(P, c, *state(mid))[1] > 0.0:
            lo = mid
        else:
            hi = mid
    ca, _, sm = state(lo)
    return c[2] * (sm - ca) >= y_min + eps * (y_c - y_min)


def _roll(case, s, kappas, rho):
    """Min slack [m, N] and its first step [m, N] of every trajectory over the whole horizon."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    N, H = case["N"], case["H"]
    d = torch.as_tensor(_disturbances(s["seed"], s["update"], N, H), device=dev)
    P = _model(s["seed"], s["update"], N, rho, dev)
    v = torch.as_tensor(s["v_prev"] + np.asarray(kappas) * (s["r"] - s["v_prev"]), device=dev).reshape(-1, 1)
    c = _consts(P, v)
    one = torch.ones((v.shape[0], N), dtype=torch.float64, device=dev)
    p_atm = P["p_atm"]
    q = [(s["x"][0] - p_atm) * one, s["x"][1] * one, (s["x"][2] - p_atm) * one]
    best = c[2] * (q[2] - q[0]) - inputs.Y_MIN
    arg = torch.zeros_like(best, dtype=torch.int64)
    for j in range(H):
        q = [a + d[i, j] for i, a in enumerate(_rk4(P, c, q))]
        slack = c[2] * (q[2] - q[0]) - inputs.Y_MIN
        less = slack < best
        best = torch.where(less, slack, best)
        arg = torch.where(less, torch.full_like(arg, j + 1), arg)
    return best, arg, d


def _gradient(case, s, kappa, d, k, j):
    """The slack of scenario k at step j and its derivatives by (kappa, x_t, parameters), by torch's autograd."""
    kap = torch.tensor(float(kappa), dtype=torch.float64, requires_grad=True)
    x = torch.tensor(s["x"], dtype=torch.float64, requires_grad=True)
    theta = torch.tensor(inputs.fc3_params(), requires_grad=True)
    P = {n: theta[i] for n, i in _NAMES.items()}
    c = _consts(P, s["v_prev"] + kap * (s["r"] - s["v_prev"]))
    q = [x[0] - P["p_atm"], x[1], x[2] - P["p_atm"]]
    dk = d[:, :, k].cpu()
    for i in range(j):
        q = [a + e for a, e in zip(_rk4(P, c, q), dk[:, i])]
    slack = c[2] * (q[2] - q[0]) - inputs.Y_MIN
    slack.backward()
    return float(slack), np.concatenate([[float(kap.grad)], x.grad.numpy(), theta.grad.numpy()])


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("eval", "gradient"):
        # the updates' results are the end points of a search (equal, or wrong); a closed loop's states would take the
        # whole search of every step in 64 bits
        return None
    s = prepare(case, seed)
    best, arg, d = _roll(case, s, s["kappas"], case.get("unc", 0.0))
    ss = np.array([_steady_ok(s["v_prev"] + k * (s["r"] - s["v_prev"])) for k in s["kappas"]])
    if kind == "eval":
        low = np.where(ss, best.min(dim=1).values.cpu().numpy(), np.nan)
        return {"admissible": None, "min_slack": low, "P": None}
    val, grad = [], []
    for i, kappa in enumerate(s["kappas"]):
        k = int(best[i].argmin())
        g, dg = _gradient(case, s, kappa, d, k, int(arg[i, k]))
        val.append(g)
        grad.append(dg)
    return {"g": np.array(val), "grad": np.array(grad), "k": None, "j": None, "ss_ok": None}
