"""What a user of this library has it do, as cases to be timed.

An inversion is created from host arrays (tau, F, sigma, omega), annealed block by block and
averaged.  The cases are whole inversions, single blocks of a long anneal (the unit that every
run repeats: sweeps, residual recomputation, branching, statistics, then the average that a run
watches), a batch of uneven inversions, and the recomputation of the residuals of given spectra.
Sizes are those of the repository's workloads: the tiny grid (32 tau x 64 bins x 64 walkers),
the paper-scale grid (200 x 1000 x 4096), the band example (160 x 1000 x 1500 walkers), the
precision workload (512 x 2048 x 16384) and the uneven batch (50-500 tau, 200-2000 bins).

The blocks run at temperatures of the order of the residue, as the first half of a schedule
does: there a decision lies further from its threshold than FP32's rounding (and its drift over
the sweeps between two recomputations) reaches, so that a block's result is a number and not a
matter of which last bit a chain of 1e8 decisions met.
"""
import math

import numpy as np
import torch

import paper_1609_07936_gb300 as sail

TWO_PI = 2.0 * math.pi


def listed():
    block = {"kind": "block", "n_sweeps": 20000, "spb": 100, "resync": 2}
    return [
        # a small data set inverted from its host arrays to its spectrum: latency and launches
        {"name": "inversion_tiny", "kind": "inversion", "n_tau": 32, "n_omega": 64, "walkers": 64, "n_sweeps": 1000,
         "spb": 100, "resync": 0, "tau_max": 4.0, "w_max": 10.0, "T_start": 1.0, "T_end": 1e-4},
        # the same in the FP64 precision mode (the one to check a result with)
        {"name": "inversion_tiny_fp64", "kind": "inversion", "n_tau": 32, "n_omega": 64, "walkers": 64,
         "n_sweeps": 200, "spb": 100, "resync": 0, "tau_max": 4.0, "w_max": 10.0, "T_start": 1.0, "T_end": 1e-4,
         "fp64": True},
        # the published problem size, whole: creation, ten blocks, average
        {"name": "inversion_paper", "kind": "inversion", "n_tau": 200, "n_omega": 1000, "walkers": 4096,
         "n_sweeps": 1000, "spb": 100, "resync": 2},
        # a block of the published schedule (T from 10 chi2_0), the default options
        {"name": "block_paper", **block, "n_tau": 200, "n_omega": 1000, "walkers": 4096},
        # a block of the schedule that reaches the noise level (absolute temperatures, finer
        # moves), part way down: fewer proposals fail the positivity test
        {"name": "block_cooled", **block, "n_tau": 200, "n_omega": 1000, "walkers": 4096, "T_start_abs": 1e12,
         "T_end_abs": 0.03, "scale": 0.1},
        # the band example: few walkers, self-cooling, adaptive branching, smoothing
        {"name": "block_band", **block, "n_tau": 160, "n_omega": 1000, "walkers": 1500, "tau_max": 7.95, "w_max": 3.5,
         "band": True, "cooling": True, "smooth": 0.01},
        # the largest: wide data, fine bins, the full population
        {"name": "block_wide", **block, "n_tau": 512, "n_omega": 2048, "walkers": 16384, "spb": 10, "peaks": 3},
        # shared bins: groups of 4 walkers move the same bins
        {"name": "block_shared", **block, "n_tau": 200, "n_omega": 1000, "walkers": 4096, "spb": 50, "shared": 4},
        # bins chosen by the index walk
        {"name": "block_walk", **block, "n_tau": 200, "n_omega": 1000, "walkers": 1500, "spb": 50, "walk": 2},
        # the Hastings-corrected move on an uneven tau grid of odd size
        {"name": "block_hastings_uneven", **block, "n_tau": 117, "n_omega": 501, "walkers": 1023, "n_sweeps": 200000,
         "spb": 50, "resync": 0, "uneven": True, "hastings": True},
        # many independent inversions side by side (one block of each)
        {"name": "batch_uneven", "kind": "batch", "problems": 12, "max_tau": 500, "max_omega": 2000,
         "max_walkers": 4096, "spb": 10, "n_sweeps": 20000, "resync": 2},
        # residuals and chi2 of spectra that the user brings (a warm start, a check)
        {"name": "residuals", "kind": "residuals", "n_tau": 200, "n_omega": 500, "walkers": 1024, "resync": 2,
         "n_sweeps": 1000, "spb": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["block", "inversion", "batch", "residuals"], [6, 2, 1, 2])[0]
    if kind == "batch":
        return {"kind": "batch", "problems": rng.randint(2, 12), "max_tau": _log(rng, 60, 500),
                "max_omega": _log(rng, 220, 2000), "max_walkers": _log(rng, 300, 4096), "spb": 10,
                "n_sweeps": 200000, "resync": rng.choice([0, 2])}
    c = {"kind": kind, "n_tau": _log(rng, 16, 512), "n_omega": _log(rng, 48, 2048), "resync": rng.choice([0, 1, 2, 2]),
         "peaks": rng.randint(1, 4), "tau_max": round(rng.uniform(3.0, 8.0), 2), "w_max": round(rng.uniform(8.0, 20.0), 2),
         "uneven": rng.random() < 0.25}
    if kind == "residuals":
        return {**c, "walkers": _log(rng, 16, 4096), "n_sweeps": 1000, "spb": 100}
    # sweeps in a block: as many as keep a pass within the largest listed case
    c["walkers"] = _log(rng, 64, 16384)
    room = 512 * 2048 * 16384 * 10 / (max(c["n_tau"], 64) * c["n_omega"] * max(c["walkers"], 1024))
    c["spb"] = max(1, min(100, int(room)))
    if kind == "inversion":
        return {**c, "n_sweeps": c["spb"] * (1 if room < 400 else 2)}
    c["n_sweeps"] = 400000
    option = rng.choice(["", "", "", "scale", "cooling", "shared", "walk", "hastings", "guard"])
    if option == "scale":
        c["scale"] = round(rng.uniform(0.05, 0.9), 3)
    elif option == "cooling":
        c["cooling"], c["smooth"] = True, rng.choice([0.0, 0.01])
    elif option == "shared":
        c["shared"] = rng.choice([2, 4, 8]) if c["n_tau"] <= 256 else rng.choice([2, 4])
    elif option == "walk":
        c["walk"], c["walkers"] = rng.randint(1, 4), min(c["walkers"], 4096)
    elif option:
        c[option] = True
    return c


def _spectrum(rng, peaks, w_max, band):
    """Peaks of a spectrum on [0, w_max] and its values on a fine grid (mass 2 pi)."""
    n = 4096
    w = (np.arange(n) + 0.5) * (w_max / n)
    S = np.zeros(n)
    if band:  # two unit Lorentzians cut to [0.5, 2.5]
        S = 1.0 / (1.0 + (w - 1.0) ** 2) + 1.0 / (1.0 + (w - 2.0) ** 2)
        S[(w < 0.5) | (w > 2.5)] = 0.0
    elif peaks == 2:  # centres 0.2 and 0.5 of 10, half widths 0.3 and 0.5
        S = 0.6 * 0.3 / ((w - 2.0) ** 2 + 0.09) + 0.4 * 0.5 / ((w - 5.0) ** 2 + 0.25)
    else:
        for c, h, a in zip(rng.uniform(0.05, 0.75, peaks) * w_max, rng.uniform(0.1, 2.0, peaks), rng.dirichlet(np.ones(peaks))):
            S += a * h / ((w - c) ** 2 + h * h)
    return w, S * (TWO_PI / (S.sum() * (w_max / n)))


def _data(case, seed):
    """Host arrays of a synthetic measurement: tau, F with noise, sigma, bin centres, A and B."""
    rng = np.random.default_rng(int(seed))
    n_tau, n_omega = case["n_tau"], case["n_omega"]
    tau_max, w_max = case.get("tau_max", 8.0), case.get("w_max", 20.0)
    u = np.arange(n_tau) / max(1, n_tau - 1)
    tau = tau_max * (u ** 1.5 if case.get("uneven") else u)
    w, S = _spectrum(rng, case.get("peaks", 2), w_max, case.get("band"))
    dv = w[1] - w[0]
    F = np.exp(-tau[:, None] * w[None, :]) @ S * (dv / TWO_PI)
    # relative noise, constant where F falls below 1e-8 of its largest value
    sigma = case.get("noise", 1e-4) * np.maximum(F, 1e-8 * F.max())
    F = F + sigma * rng.standard_normal(n_tau)
    dw = w_max / n_omega
    omega = (np.arange(n_omega) + 0.5) * dw
    return tau, F, sigma, omega, S.sum() * dv / dw, (S * w).sum() * dv / dw


def _params(case, seed, A, B):
    p = sail.Params(n_walkers=case["walkers"], n_sweeps=case["n_sweeps"], sweeps_per_block=case["spb"],
                    resync_every=min(50, case["spb"]), resync_kind=case["resync"], A=A, B=B, seed=int(seed))
    if case.get("fp64"):
        p.precision = sail.PREC_FP64
    for key in ("T_start", "T_end", "T_start_abs", "T_end_abs"):
        if key in case:
            setattr(p, key, case[key])
    if "scale" in case:
        p.move_scale = case["scale"] / case["n_omega"]
    if case.get("cooling"):
        p.schedule_kind, p.adaptive_branching, p.smooth_s = sail.SCHEDULE_SELF_COOLING, True, case["smooth"]
    p.shared_bins = case.get("shared", 0)
    p.index_walk_len = case.get("walk", 0)
    p.hastings = bool(case.get("hastings"))
    p.fp64_accept = 1 if case.get("guard") else 0
    return p


def _uneven(case):
    """The batch's problems as cases: sizes over the whole range."""
    rng = np.random.default_rng([77, case["problems"]])
    got = []
    for k in range(case["problems"]):
        size = {"n_tau": int(rng.integers(50, case["max_tau"] + 1)), "n_omega": int(rng.integers(200, case["max_omega"] + 1)),
                "walkers": int(rng.integers(256, case["max_walkers"] + 1)), "peaks": int(rng.integers(1, 5)),
                "noise": float(10.0 ** rng.uniform(-5, -3))}
        got.append({"kind": "block", "n_sweeps": case["n_sweeps"], "spb": case["spb"], "resync": case["resync"], **size})
    return got


def prepare(case, seed):
    if case["kind"] == "batch":
        problems = []
        for k, c in enumerate(_uneven(case)):
            *arrays, A, B = _data(c, int(seed) * 64 + k)
            problems.append((*arrays, _params(c, int(seed) * 64 + k, A, B)))
        return {"case": case, "batch": sail.Batch(problems)}
    *arrays, A, B = _data(case, seed)
    state = {"case": case, "arrays": arrays, "params": _params(case, seed, A, B)}
    if case["kind"] != "inversion":
        state["sail"] = sail.Sail(*arrays, state["params"])
    if case["kind"] == "residuals":
        state["a"] = _spectra(case, seed, A)
    return state


def _spectra(case, seed, A):
    """Spectra of the right mass: smooth densities with a spread of shapes."""
    rng = np.random.default_rng(int(seed) + 1)
    x = (np.arange(case["n_omega"]) + 0.5) / case["n_omega"]
    c, h = rng.uniform(0.05, 0.6, (case["walkers"], 1)), rng.uniform(0.02, 0.3, (case["walkers"], 1))
    a = np.exp(-0.5 * ((x - c) / h) ** 2) + 0.05
    return a * (A / a.sum(1, keepdims=True))


def run(state):
    case = state["case"]
    if case["kind"] == "inversion":
        s = sail.Sail(*state["arrays"], state["params"])
        s.anneal()
        mean, err, used, c2 = s.average()
        s.close()
        if not case.get("fp64"):
            mean, err, c2 = mean.astype(np.float32), err.astype(np.float32), np.float32(c2)
        return {"mean": mean, "err": err, "used": used, "chi2_of_mean": c2}
    if case["kind"] == "batch":
        state["batch"].anneal(1)
        return [_averaged(s) for s in state["batch"].handles]
    s = state["sail"]
    if case["kind"] == "residuals":
        s.set_state(state["a"])
        _, R, chi2, _, _ = s.state()
        return {"R": R.astype(np.float32), "chi2": chi2.astype(np.float32)}
    s.anneal(1)
    a, R = s.walker_rows(np.arange(case["walkers"]))
    return {**_averaged(s), "a": a.float(), "R": R.float()}


def _averaged(s):
    """What a run watches; an FP32 handle's values as floats, which is what they come from."""
    mean, err, used, c2 = s.average()
    return {"mean": mean.astype(np.float32), "err": err.astype(np.float32), "used": used, "chi2_of_mean": np.float32(c2),
            "chi2": s.chi2().astype(np.float32)}


# A move changes the residual within the span of the kernel's columns.  The Laplace kernel's
# numerical rank at FP32 is about 24, whatever the number of tau points, so a move cannot do
# without 9 operations (the change from three vectors, its product with the residual) on each
# of that many directions; a proposal that fails the positivity test (0.4 of them) needs none.
RANK, OPS, FEASIBLE = 24, 9, 0.6


def work(case):
    if case["kind"] == "batch":
        parts = [work(c) for c in _uneven(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n_tau, n_omega, W = case["n_tau"], case["n_omega"], case["walkers"]
    word = 8 if case.get("fp64") else 4
    if case["kind"] == "residuals":  # host spectra in (FP64), residuals and spectra out
        return {"bytes": 8.0 * W * (2 * n_omega + n_tau + 1), "flops": 2.0 * W * n_tau * n_omega}
    sweeps = case["n_sweeps"] if case["kind"] == "inversion" else case["spb"]
    moves = float(sweeps) * W * n_omega
    recomputed = 2.0 * W * n_tau * n_omega * -(-sweeps // min(50, case["spb"]))
    return {"bytes": word * W * (2.0 * n_omega + 2.0 * n_tau) + 8.0 * (3 * n_tau + n_omega),
            "flops": moves * FEASIBLE * OPS * min(n_tau, RANK) + recomputed}


def exact(case, seed):
    """The residuals in 64 bits.  An anneal's result is a draw from a chain and has no such value."""
    if case["kind"] != "residuals":
        return None
    tau, F, sigma, omega, A, B = _data(case, seed)
    a = _spectra(case, seed, A)
    dw = (omega[-1] - omega[0]) / (omega.size - 1)
    j, t = np.arange(omega.size)[None, :], tau[:, None]
    with np.errstate(divide="ignore", invalid="ignore"):
        K = np.where(t == 0.0, dw / TWO_PI, np.exp(-j * dw * t) * -np.expm1(-dw * t) / (TWO_PI * t))
    R = F / sigma - a @ (K / sigma[:, None]).T
    return {"R": R, "chi2": (R * R).sum(1)}
