"""The work that a user of the library has it do, as cases that can be timed one by one.

Each case is one pass through the public entry points of
paper_2206_11234_gb300.native, over the sizes of the paper's runs, of the
workloads in workloads.py, of the tests and of bench.py:

  simulate   one parameter set through fpt_simulate (the README's first call)
  batch      one or several sets through fpt_simulate_batch, with histograms
  plan       several sets through a graph-captured plan, with histograms
  host       several sets through the host-buffer call, records and histograms
             copied to pinned memory
  power      one p of the power-law bias search: fpt_simulate, then fpt_pearson
  records    analysis of records in hand: fpt_histogram with jackknife subsets,
             then fpt_estimate
  network    the learned bias as a function: fpt_mlp_forward and fpt_mlp_backward
  learned    fpt_simulate_mlp, the inference of the learned bias
  train      one MlpTrainer.step from a checkpoint

The random streams are the library's own (seeded), so a simulation's input is
its parameter sets and its seed.
"""
import math

import numpy as np
import torch

from paper_2206_11234_gb300 import native as nat
from paper_2206_11234_gb300 import power_bias
from paper_2206_11234_gb300 import workloads as W

INF = 1.0e300  # "no wall" in a case (cases hold plain finite values)
C0 = 1.0 / (2.0 * math.pi * math.sqrt(6.0))
R42 = math.sqrt(42.0)


def listed():
    return [
        # A first look at a parameter set: a few hundred short runs.  Launch
        # latency and the length of the longest run are all there is.
        {"name": "pilot", "kind": "simulate", "precision": "f32_kahan", "n": 512, "phi_in": 3.0, "phi_uv": INF,
         "m": 1.0, "b": 1.0, "dN": 1e-3, "n_max": 6.0},
        # The binary64 mode at the size of workloads.quadratic_fixed_b.
        {"name": "binary64", "kind": "batch", "precision": "f64", "n": 16384, "phi_in": 3.0, "phi_uv": INF,
         "m": 1.0, "dN": 1e-3, "n_max": 6.0, "biases": "1", "n_bins": 100, "lo": 0.0, "hi": 6.0},
        # One of the paper's diffusion-dominated figures: 2e5 runs per bias, wall at the start.
        {"name": "figure", "kind": "batch", "precision": "f32_f64acc", "n": 200000, "phi_in": R42, "phi_uv": R42,
         "m": 1.0, "dN": 1e-3, "n_max": 30.0, "biases": "0,0.4,0.8", "n_bins": 60, "lo": 0.0, "hi": 30.0},
        # One p of the power-law bias search at the paper's 4e4 runs.
        {"name": "power", "kind": "power", "precision": "f32_f64acc", "n": 40000, "phi_in": 6.0, "m": 0.001,
         "p": 3.0, "sigmas": 8.0},
        # A potential other than the quadratic one: phi^4 with a wall, as in the tests, odd size.
        {"name": "quartic", "kind": "simulate", "precision": "f32_kahan", "n": 100003, "phi_in": 4.0, "phi_uv": 4.6,
         "phi_end": math.sqrt(8.0), "m": 0.0, "c4": 0.0125, "b": 0.8, "dN": 1e-3, "n_max": 40.0},
        # A scan of 64 unequal sets (workloads.batched_uneven) at 2^14 runs per set.
        {"name": "scan", "kind": "plan", "precision": "f32_kahan", "workload": "uneven", "n": 16384, "block_dim": 0,
         "k_steps": 0},
        # The headline workload: the drift-dominated bias ladder at its full size and tuned launch shape.
        {"name": "ladder", "kind": "plan", "precision": "f32_kahan", "workload": "ladder", "n": 4194304,
         "block_dim": 512, "k_steps": 64},
        # Far-tail production with host buffers (workloads.diffusion_wall), 2^16 runs per bias.
        {"name": "wall_host", "kind": "host", "precision": "f32_f64acc", "workload": "wall", "n": 65536,
         "block_dim": 0, "k_steps": 0},
        # Analysis of records in hand: jackknife histogram and per-bin estimates.
        {"name": "records", "kind": "records", "n": 16777216, "n_bins": 400, "n_sub": 10, "lo": 7.0, "hi": 10.0,
         "mean": 8.5, "sigma": 0.02, "slope": 40.0, "scatter": 2.0, "censored": 0.0},
        # The learned bias as a function of the state, with its gradient.
        {"name": "network", "kind": "network", "n": 1000003},
        # Inference with the learned bias (bench.py's learned workload at 2^18 runs).
        {"name": "learned", "kind": "learned", "n": 262144, "k_eval": 64, "b0": 0.4},
        # One Adam step of the learned bias at the bench's 2^14 runs.
        {"name": "train", "kind": "train", "n": 16384, "k_eval": 32, "b0": 0.4},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _count(rng, lo, hi):
    """A size between lo and hi, spread over its logarithm, mostly not a round one."""
    n = int(_log(rng, lo, hi))
    return max(int(lo), n - n % 1024) if n > 4096 and rng.random() < 0.25 else n


def draw(rng):
    kind = rng.choice(["simulate", "simulate", "batch", "batch64", "power", "quartic", "scan", "ladder", "host",
                       "records", "records", "network", "learned", "train"])
    if kind in ("simulate", "batch", "batch64"):
        m = rng.choice([0.01, 0.1, 1.0])
        phi_in = rng.uniform(2.0, 8.0)
        n_max = float(math.ceil(2.0 * (phi_in ** 2 - 2.0) / 4.0 + 5.0))
        wall = rng.choice([INF, phi_in, 1.2 * phi_in])
        dN = rng.choice([1e-3, 5e-4, 2e-3])
        b = rng.choice([0.0, 0.4, 0.8, 1.0, 2.0])
        if kind == "batch64":
            return {"kind": "batch", "precision": "f64", "n": _count(rng, 100, 20000), "phi_in": min(phi_in, 4.0),
                    "phi_uv": INF if wall == INF else max(wall, 4.0), "m": m, "dN": 1e-3, "n_max": 10.0,
                    "biases": "%g" % b, "n_bins": rng.choice([50, 100, 333]), "lo": 0.0, "hi": 10.0}
        prec = rng.choice(["f32_kahan", "f32_f64acc"])
        c = {"precision": prec, "phi_in": phi_in, "phi_uv": wall, "m": m, "dN": dN, "n_max": n_max}
        if kind == "simulate":
            return dict(c, kind="simulate", n=_count(rng, 64, 400000), b=b)
        return dict(c, kind="batch", n=_count(rng, 1000, 400000), biases=rng.choice(["0", "0,0.4,0.8", "0,1,2,4"]),
                    n_bins=rng.choice([60, 100, 400]), lo=0.0, hi=n_max)
    if kind == "power":
        return {"kind": "power", "precision": rng.choice(["f32_kahan", "f32_f64acc"]), "n": _count(rng, 2000, 300000),
                "phi_in": rng.uniform(4.0, 6.0), "m": 0.001, "p": rng.choice([0.0, 1.0, 2.0, 2.5, 3.0, 3.5, 4.0]),
                "sigmas": rng.choice([4.0, 8.0])}
    if kind == "quartic":
        phi_in = rng.uniform(3.2, 4.5)
        return {"kind": "simulate", "precision": rng.choice(["f32_kahan", "f32_f64acc"]), "n": _count(rng, 500, 400000),
                "phi_in": phi_in, "phi_uv": rng.choice([INF, 1.15 * phi_in]), "phi_end": math.sqrt(8.0), "m": 0.0,
                "c4": 0.0125, "b": rng.choice([0.0, 0.8]), "dN": 1e-3, "n_max": 40.0}
    if kind == "scan":
        return {"kind": "plan", "precision": "f32_kahan", "workload": "uneven", "n": _count(rng, 500, 50000),
                "block_dim": 0, "k_steps": 0}
    if kind == "ladder":
        return {"kind": "plan", "precision": rng.choice(["f32_kahan", "f32_f64acc"]), "workload": "ladder",
                "n": _count(rng, 5000, 3000000), "block_dim": 512, "k_steps": 64}
    if kind == "host":
        return {"kind": "host", "precision": "f32_f64acc", "workload": rng.choice(["wall", "ladder"]),
                "n": _count(rng, 2000, 200000), "block_dim": 0, "k_steps": 0}
    if kind == "records":
        n_bins, n_sub = rng.choice([(400, 1), (400, 10), (60, 16), (40, 16), (512, 1), (4095, 1), (200, 20)])
        return {"kind": "records", "n": _count(rng, 1000, 20000000), "n_bins": n_bins, "n_sub": n_sub, "lo": 7.0,
                "hi": 10.0, "mean": 8.5, "sigma": rng.choice([0.02, 0.1, 0.5]), "slope": rng.choice([0.0, 5.0, 40.0]),
                "scatter": rng.choice([0.0, 0.5, 2.0]), "censored": rng.choice([0.0, 0.02])}
    if kind == "network":
        return {"kind": "network", "n": _count(rng, 100, 4000000)}
    if kind == "learned":
        return {"kind": "learned", "n": _count(rng, 1000, 262144), "k_eval": rng.choice([32, 64, 128]),
                "b0": rng.uniform(0.2, 0.5)}
    return {"kind": "train", "n": _count(rng, 1024, 16384), "k_eval": rng.choice([32, 64]), "b0": rng.uniform(0.2, 0.5)}


# ---- what a user's program has in hand before the call ----

def _wall(x):
    return math.inf if x >= INF else x


def _specs(case):
    """The parameter sets of a batch, plan or host case."""
    if case["kind"] == "batch":
        return [W.SetSpec(phi_in=case["phi_in"], m=case["m"], b=float(b), dN=case["dN"], n_max=case["n_max"],
                          n_traj=case["n"], phi_uv=_wall(case["phi_uv"]), set_id=i, hist_lo=case["lo"],
                          hist_hi=case["hi"], n_bins=case["n_bins"])
                for i, b in enumerate(case["biases"].split(","))]
    wl = {"uneven": W.batched_uneven, "ladder": W.drift_dominated_ladder, "wall": W.diffusion_wall}[case["workload"]]()
    for s in wl.sets:
        s.n_traj = case["n"]
    return wl.sets


NORM = (5.2, 0.5, 30.0, 1.0 / 15.0)  # input normalisation of the learned-bias workload


def _net(b0, gain=1.0, out_scale=0.05, seed=5):
    p = W.mlp_params(seed=seed, gain=gain, out_scale=out_scale)
    p[-1] = b0
    return p


def _records(case, seed):
    """(N, ln w) as a biased run leaves them: N normal about its mean, ln w falling with N plus a scatter."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn(case["n"], generator=g, dtype=torch.float64, device="cuda")
    N = case["mean"] + case["sigma"] * z
    lw = torch.randn(case["n"], generator=g, dtype=torch.float64, device="cuda")
    lw = -case["slope"] * (N - case["mean"]) + case["scatter"] * lw - 3.0
    if case["censored"] > 0.0:
        u = torch.rand(case["n"], generator=g, dtype=torch.float64, device="cuda")
        N = torch.where(u < case["censored"], torch.full_like(N, math.inf), N)
    return N, lw


def _rows(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(case["n"], generator=g, dtype=torch.float32, device="cuda")
    v = torch.rand(case["n"], generator=g, dtype=torch.float32, device="cuda")
    # states of the learned workload: phi between phi_end and the wall, N up to the cap
    return 1.42 + 7.58 * u, 60.0 * v, torch.randn(case["n"], generator=g, dtype=torch.float32, device="cuda") / case["n"]


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    f64 = dict(dtype=torch.float64, device="cuda")
    s = {"case": case, "seed": seed}
    if kind == "simulate":
        model = dict(model=nat.MODEL_POLYNOMIAL, poly=[0.0, 0.0, 0.0, 0.0, case["c4"]]) if "c4" in case else {}
        s["params"] = nat.make_params(precision=case["precision"], m=case["m"], n_max=case["n_max"], **model)
        s["N"], s["lw"] = torch.empty(n, **f64), torch.empty(n, **f64)
    elif kind in ("batch", "plan", "host"):
        specs = _specs(case)
        total = sum(x.n_traj for x in specs)
        s["sets"] = nat.make_sets(specs)
        s["params"] = nat.make_params(precision=case["precision"], m=specs[0].m, n_max=specs[0].n_max,
                                      block_dim=case.get("block_dim", 0), k_steps=case.get("k_steps", 0))
        if kind == "host":
            f = dict(dtype=torch.float64, pin_memory=True)
            s["N"], s["lw"] = torch.empty(total, **f), torch.empty(total, **f)
            s["bins"] = torch.empty((sum(x.n_bins for x in specs), nat.BIN_FIELDS), **f)
            s["counts"] = torch.empty((len(specs), 4), dtype=torch.int64, pin_memory=True)
        else:
            s["N"], s["lw"] = torch.empty(total, **f64), torch.empty(total, **f64)
            s["bins"], s["counts"] = nat.empty_bins(sum(x.n_bins for x in specs)), nat.empty_counts(len(specs))
        if kind == "plan":
            s["plan"] = nat.Plan(s["params"], s["sets"], s["N"], s["lw"], s["bins"], s["counts"])
    elif kind == "power":
        sigma = power_bias.classical_sigma(case["m"], case["phi_in"])
        target = (case["phi_in"] ** 2 - 2.0) / 4.0 + case["sigmas"] * sigma
        s["amp"] = power_bias.tune_amplitude(case["p"], target, case["phi_in"])
        s["dN"] = sigma / 20.0
        s["params"] = nat.make_params(precision=case["precision"], m=case["m"], n_max=target + 40.0 * sigma,
                                      bias_p=case["p"])
        s["N"], s["lw"], s["out"] = torch.empty(n, **f64), torch.empty(n, **f64), torch.empty(8, **f64)
    elif kind == "records":
        s["N"], s["lw"] = _records(case, seed)
        s["bins"], s["counts"] = nat.empty_bins(case["n_bins"] * case["n_sub"]), nat.empty_counts(1)
        s["est"] = nat.empty_estimates(case["n_bins"])
    elif kind == "network":
        s["w"] = nat.mlp_pack(_net(0.0, gain=1.5, out_scale=1.0, seed=11), NORM)
        s["phi"], s["Nin"], s["g"] = _rows(case, seed)
        s["b"] = torch.empty(n, dtype=torch.float32, device="cuda")
        s["grad"] = torch.empty(nat.MLP_NPARAM, dtype=torch.float32, device="cuda")
    elif kind == "learned":
        spec = W.SetSpec(phi_in=8.0, m=1.0, b=0.0, dN=5e-4, n_max=60.0, phi_uv=9.0, n_traj=n)
        s["w"] = nat.mlp_pack(_net(case["b0"]), NORM)
        s["sets"] = nat.make_sets([spec])
        s["params"] = nat.make_params(precision="f32_f64acc", m=1.0, n_max=60.0, mlp=s["w"], k_eval=case["k_eval"])
        s["N"], s["lw"] = torch.empty(n, **f64), torch.empty(n, **f64)
    else:
        spec = W.SetSpec(phi_in=8.0, m=1.0, b=0.0, dN=5e-4, n_max=60.0, phi_uv=9.0, n_traj=n)
        t = nat.MlpTrainer(spec, _net(case["b0"]), NORM, k_eval=case["k_eval"])
        s["trainer"] = t
        s["checkpoint"] = [(x, x.clone()) for x in (t.master, t.adam_m, t.adam_v, t.w)]
    return s


# ---- one pass ----

def _bins_out(bins, counts):
    return {"max_lw": bins[:, 0], "sums": bins[:, 1:3], "moments": bins[:, 3:7], "count": bins.view(torch.int64)[:, 7],
            "counts": counts}


def run(s):
    case, seed = s["case"], s["seed"]
    kind, n = case["kind"], case["n"]
    if kind == "simulate":
        nat.fpt_simulate(s["params"], n, case["phi_in"], case.get("phi_end", W.PHI_END), _wall(case["phi_uv"]),
                         case["dN"], case["b"], seed, s["N"], s["lw"])
        return {"N": s["N"], "lw": s["lw"]}
    if kind == "batch":
        nat.fpt_simulate_batch(s["params"], s["sets"], seed, s["N"], s["lw"], s["bins"], s["counts"])
        return dict(_bins_out(s["bins"], s["counts"]), N=s["N"], lw=s["lw"])
    if kind == "plan":
        s["plan"].launch(seed)
        return dict(_bins_out(s["bins"], s["counts"]), N=s["N"], lw=s["lw"])
    if kind == "host":
        nat.fpt_simulate_batch_host(s["params"], s["sets"], seed, s["N"], s["lw"], s["bins"], s["counts"])
        return dict(_bins_out(s["bins"], s["counts"]), N=s["N"], lw=s["lw"])
    if kind == "power":
        nat.fpt_simulate(s["params"], n, case["phi_in"], W.PHI_END, math.inf, s["dN"], s["amp"], seed, s["N"], s["lw"])
        r = nat.fpt_pearson(s["N"], s["lw"], s["out"])
        return {"N": s["N"], "lw": s["lw"], "pearson": [r[f] for f in nat.PEARSON_FIELDS]}
    if kind == "records":
        nat.fpt_histogram(s["N"], s["lw"], case["n_bins"], case["lo"], case["hi"], s["bins"], s["counts"],
                          n_sub=case["n_sub"])
        nat.fpt_estimate(s["bins"], case["n_bins"], case["lo"], case["hi"], n, s["est"], n_sub=case["n_sub"])
        return dict(_bins_out(s["bins"], s["counts"]), estimates=s["est"])
    if kind == "network":
        nat.fpt_mlp_forward(s["w"], s["phi"], s["Nin"], s["b"])
        s["grad"].zero_()
        nat.fpt_mlp_backward(s["w"], s["phi"], s["Nin"], s["g"], s["grad"])
        return {"b": s["b"], "grad": s["grad"]}
    if kind == "learned":
        nat.fpt_simulate_mlp(s["params"], s["sets"], seed, s["N"], s["lw"])
        return {"N": s["N"], "lw": s["lw"]}
    t = s["trainer"]
    for x, y in s["checkpoint"]:
        x.copy_(y)
    t.state.step = 0
    stats = t.step(seed=seed, tail_N=40.0, lr=3e-3)
    return {"grad": t.grad, "master": t.master, "adam_m": t.adam_m, "adam_v": t.adam_v, "N": t.out_N,
            "lw": t.out_logw, "n_records": stats["n_records"], "log_second_moment": stats["log_second_moment"]}


# ---- the work of one pass ----

def _duration(phi_in, m, b, n_max, phi_end=W.PHI_END):
    """The noise-free duration of a run of the quadratic model with drift -2/phi + b C0 m phi, at most n_max."""
    k = b * C0 * m
    if k <= 0.0:
        return min(n_max, (phi_in ** 2 - phi_end ** 2) / 4.0)
    if k * phi_in ** 2 >= 2.0:
        return n_max
    return min(n_max, math.log((2.0 - k * phi_end ** 2) / (2.0 - k * phi_in ** 2)) / (2.0 * k))


# One Euler–Maruyama step: 11 integer operations of Philox4x32-10 (three
# counters of 60 per 16 steps), 6 of half a Box–Muller pair, 7 of the update,
# the weight sum and the wall.
STEP_OPS = 24.0
ROW_FLOPS = 2.0 * nat.MLP_NPARAM  # one evaluation of the network


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "records":
        return {"bytes": 16.0 * n + 64.0 * case["n_bins"] * case["n_sub"] + 144.0 * case["n_bins"], "flops": 24.0 * n}
    if kind == "network":
        return {"bytes": 24.0 * n, "flops": 4.0 * ROW_FLOPS * n}
    if kind in ("learned", "train"):
        steps = n * 16.0 / 5e-4  # the mean duration of these runs is about 16
        flops = steps * STEP_OPS + (steps / case["k_eval"]) * ROW_FLOPS * (1.0 if kind == "learned" else 2.0)
        return {"bytes": 16.0 * n, "flops": flops}
    if kind == "power":
        sigma = power_bias.classical_sigma(case["m"], case["phi_in"])
        steps = n * ((case["phi_in"] ** 2 - 2.0) / 4.0 + case["sigmas"] * sigma) / (sigma / 20.0)
        return {"bytes": 32.0 * n, "flops": steps * (STEP_OPS + 6.0)}
    if kind == "simulate":
        if "c4" in case:
            d = min(case["n_max"], (case["phi_in"] ** 2 - case["phi_end"] ** 2) / 8.0)
        else:
            d = _duration(case["phi_in"], case["m"], case["b"], case["n_max"])
        return {"bytes": 16.0 * n, "flops": n * d / case["dN"] * STEP_OPS}
    specs = _specs(case)
    steps = sum(x.n_traj * _duration(x.phi_in, x.m, x.b, x.n_max) / x.dN for x in specs)
    return {"bytes": sum(32.0 * x.n_traj + 64.0 * x.n_bins for x in specs), "flops": steps * STEP_OPS}


# ---- the same results in 64 bits, by plain torch ----

M32 = 0xFFFFFFFF


def _mulhilo(a, x):
    """(high, low) 32 bits of a * x for a constant a < 2^32 and int64 tensors x < 2^32."""
    lo = a * (x & 0xFFFF)
    hi = a * (x >> 16) + (lo >> 16)
    return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)


def _philox(c0, ident, set_id, seed):
    """Philox4x32-10 of the counters (c0, ident, 0, set_id): four int64 tensors."""
    x0, x1, x2, x3 = c0 + 0 * ident, ident + 0 * c0, 0 * (c0 + ident), set_id + 0 * (c0 + ident)
    k0, k1 = seed & M32, seed >> 32
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, x0)
        h1, l1 = _mulhilo(0xCD9E8D57, x2)
        x0, x1, x2, x3 = h1 ^ x1 ^ k0, l1, h0 ^ x3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x0, x1, x2, x3


def _simulate64(n, set_id, seed, bits, phi_in, phi_end, phi_uv, m, b, dN, n_max):
    """(N, ln w) of the quadratic model with a constant bias, binary64; `bits`: the radius word's bits in use."""
    ident = torch.arange(n, dtype=torch.int64, device="cuda")
    phi = torch.full((n,), phi_in, dtype=torch.float64, device="cuda")
    N = torch.full_like(phi, math.inf)
    Wsum, steps, live = torch.zeros_like(phi), torch.zeros_like(phi), torch.ones_like(ident, dtype=torch.bool)
    cm, sq, m_max = C0 * m, math.sqrt(dN), math.ceil(n_max / dN)
    k = 0
    while k < m_max and bool(live.any()):
        V = [w for j in range(3) for w in _philox(torch.full_like(ident, 3 * (k // 16) + j), ident, set_id, seed)]
        for j in range(4):
            for p in range(2):
                rad, ang = V[3 * j + p], (V[3 * j + 2] >> 16) if p == 0 else (V[3 * j + 2] & 0xFFFF)
                u0 = ((rad >> (32 - bits)).double() + 0.5) * 2.0 ** -bits
                r, a = torch.sqrt(-2.0 * torch.log(u0)), 2.0 * math.pi * ((ang.double() + 0.5) * 2.0 ** -16)
                for xi in (r * torch.cos(a), r * torch.sin(a)):
                    if k >= m_max:
                        continue
                    new = phi + (-2.0 / phi + b * (cm * phi)) * dN + cm * phi * xi * sq
                    if phi_uv < INF:
                        new = torch.minimum(new, 2.0 * phi_uv - new)
                    hit = live & (new <= phi_end)
                    N = torch.where(hit, (k + (phi - phi_end) / (phi - new)) * dN, N)
                    Wsum = torch.where(live, Wsum + xi, Wsum)
                    steps = torch.where(live, steps + 1.0, steps)
                    live = live & ~hit
                    phi = torch.where(live, new, phi)
                    k += 1
    return N, -b * sq * Wsum - 0.5 * b * b * dN * steps


def _histogram64(N, lw, n_bins, n_sub, lo, hi):
    d = (hi - lo) / n_bins
    ok = torch.isfinite(N) & (N > lo) & (N <= hi)
    sub = torch.arange(N.numel(), device=N.device) % n_sub
    j = torch.where(ok, torch.clamp(torch.ceil((N - lo) / d) - 1.0, 0, n_bins - 1), torch.zeros_like(N)).long()
    at = (sub * n_bins + j)[ok]
    x = lw[ok]
    nb = n_bins * n_sub
    mx = torch.full((nb,), -math.inf, dtype=torch.float64, device=N.device).scatter_reduce(0, at, x, "amax")
    x = x - mx[at]
    e = torch.exp(x)
    s = [torch.zeros(nb, dtype=torch.float64, device=N.device).index_add_(0, at, y)
         for y in (e, e * e, x, x * x, x ** 3, x ** 4)]
    return mx, torch.stack(s[:2], 1), torch.stack(s[2:], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("simulate", "batch"):
        # a step at a time over all runs: only where that is quick
        if "c4" in case or case["n"] > 20000 or case["n_max"] / case["dN"] > 12000:
            return None
        bits = 32 if case["precision"] == "f64" else 23
        args = (case["phi_in"], W.PHI_END, case["phi_uv"], case["m"])
        if kind == "simulate":
            N, lw = _simulate64(case["n"], 0, seed, bits, *args, case["b"], case["dN"], case["n_max"])
            return {"N": N, "lw": lw}
        b = case["biases"].split(",")
        if len(b) > 1:
            return None
        N, lw = _simulate64(case["n"], 0, seed, bits, *args, float(b[0]), case["dN"], case["n_max"])
        mx, sums, moments = _histogram64(N, lw, case["n_bins"], 1, case["lo"], case["hi"])
        return {"N": N, "lw": lw, "max_lw": mx, "sums": sums, "moments": moments, "count": None, "counts": None}
    if kind == "records":
        N, lw = _records(case, seed)
        mx, sums, moments = _histogram64(N, lw, case["n_bins"], case["n_sub"], case["lo"], case["hi"])
        return {"max_lw": mx, "sums": sums, "moments": moments, "count": None, "counts": None, "estimates": None}
    if kind == "network":
        p = _net(0.0, gain=1.5, out_scale=1.0, seed=11)
        p = torch.as_tensor(np.asarray(p), dtype=torch.float32).to(torch.bfloat16).double().cuda().requires_grad_(True)
        h = nat.MLP_HIDDEN
        phi, Nin, g = (x.double() for x in _rows(case, seed))
        norm = torch.tensor(NORM, dtype=torch.float32).double()
        b = torch.empty_like(phi)
        for i in range(0, phi.numel(), 1 << 18):
            x = torch.stack([(phi[i:i + (1 << 18)] - norm[0]) * norm[1], (Nin[i:i + (1 << 18)] - norm[2]) * norm[3]], 1)
            h1 = torch.tanh(x @ p[:2 * h].view(h, 2).T + p[2 * h:3 * h])
            h2 = torch.tanh(h1 @ p[3 * h:3 * h + h * h].view(h, h).T + p[3 * h + h * h:4 * h + h * h])
            y = h2 @ p[4 * h + h * h:5 * h + h * h] + p[5 * h + h * h]
            b[i:i + (1 << 18)] = y.detach()
            (y * g[i:i + (1 << 18)]).sum().backward()
        return {"b": b, "grad": p.grad}
    return None
