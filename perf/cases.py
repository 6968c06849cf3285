"""The work that a user of this framework has it do, as measurable cases.

Kinds of case, each through the package's public entry points:

  run     one parameter point: Engine.run and Engine.stats, with per-path outputs
  scan    many parameter points in one call: Engine.scan (statistics on the
          host) or Engine.scan_device (sums left on the device)
  chi     the step-size probe: Engine.local_error
  forward the surrogate network's predictions: Surrogate.forward
  screen  the guided scan's screen of a grid: guided.predict with two networks
          and guided.select
  fit     training on labels: Surrogate.fit, then Surrogate.get_params
  train   a training loop of the caller's own: Surrogate.train_step per batch,
          then Surrogate.get_params

Parameter values, step sizes and path counts are those of
paper_1409_4923_gb300.workloads, of the paper's validation settings and of the
tests; horizons are cut so that a pass stays well below a second (the work of a
run is proportional to its horizon).  Everything follows from the seed alone.

exact() gives the value of a case in 64 bits where it has one.  The driven
inertial washboard is chaotic: beyond one drive period two roundings of the same
path part, so the inertial runs and scans have no such value; nor have the
weights after many Adam steps, whose first steps are the signs of gradients.
"""
import math

import numpy as np
import torch

from paper_1409_4923_gb300 import engine, guided, surrogate, workloads

OMEGA = 4.9
GAUSS, POISSON, DICHOT, NORMAL, COMPENSATED = 1, 2, 4, 8, 16


def listed():
    return [
        # The Poisson workload as it stands (100 + 400 drive periods): one
        # parameter point at the paper's ensemble size, the smallest useful
        # run; a path per lane on a nearly idle GPU, so latency per step counts.
        {"name": "run_poisson_1024", "kind": "run", "what": "poisson", "paths": 1024, "spp": 100,
         "transient": 100, "periods": 400, "block": 128, "ppt": 1},
        # The 2^20-path dichotomous ensemble with the tuned launch shape: the
        # throughput of the step loop on a full GPU.
        {"name": "run_dichot_2p20", "kind": "run", "what": "dichot", "paths": 1 << 20, "spp": 200,
         "transient": 20, "periods": 80, "block": 64, "ppt": 2},
        # The paper's validation run of Model I (overdamped, piecewise-linear
        # potential, Poissonian noise alone): 1024 paths, 400 steps per
        # 1 / lambda, launches of 4000 steps with the states kept in between.
        {"name": "run_model1_1024", "kind": "run", "what": "model1", "paths": 1024, "spp": 400,
         "transient": 10, "periods": 90, "block": 128, "ppt": 1, "samples": 4000},
        # Gaussian increments by Box-Muller and the compensated Poisson bias,
        # an odd path count and ragged step counts, the default launch shape.
        {"name": "run_normal_20011", "kind": "run", "what": "normal", "paths": 20011, "spp": 97,
         "transient": 5, "periods": 45, "block": 128, "ppt": 1},
        # Every 16th point of the 64 x 64 Poisson scan, uneven paths and
        # horizons: a map of <v>(F, Q) at plain Monte Carlo.
        {"name": "scan_poisson_256", "kind": "scan", "what": "poisson", "points": 256, "paths_lo": 256,
         "paths_hi": 16384, "spp": 100, "transient": 10, "periods_lo": 50, "periods_hi": 300, "device": False},
        # Many points of few paths: a coarse map, one persistent launch.
        {"name": "scan_small_points", "kind": "scan", "what": "poisson", "points": 512, "paths_lo": 32,
         "paths_hi": 1024, "spp": 100, "transient": 10, "periods_lo": 50, "periods_hi": 150, "device": False},
        # The guided scan's labels: points of the dichotomous model at 2048
        # paths each, results left on the device.
        {"name": "scan_dichot_labels", "kind": "scan", "what": "dichot", "points": 512, "paths_lo": 2048,
         "paths_hi": 2048, "spp": 200, "transient": 10, "periods_lo": 100, "periods_hi": 100, "device": True},
        # A probe of the step-size control: 4096 paths over one drive period.
        {"name": "chi_4096", "kind": "chi", "what": "poisson", "paths": 4096, "spp": 100, "steps": 100},
        # Predictions for the points of a 64 x 64 scan.
        {"name": "forward_4096", "kind": "forward", "rows": 4096},
        # The guided scan's screen of its 1024 x 1024 grid.
        {"name": "screen_1024x1024", "kind": "screen", "nx": 1024, "ny": 1024},
        # The guided scan's training (batch 512 of 8192 labels), 200 of its steps.
        {"name": "fit_512_of_8192", "kind": "fit", "labels": 8192, "batch": 512, "steps": 200},
        # A large-batch training loop of the caller's own.
        {"name": "train_16384", "kind": "train", "rows": 16384, "steps": 4},
    ]


def _between(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "scan", "scan", "chi", "forward", "screen", "fit", "train"])
    if kind == "run":
        what = rng.choice(["poisson", "dichot", "model1", "normal", "both", "washboard"])
        paths = _between(rng, 32, 1 << 20)
        steps = max(500, min(50000, int(1.5e10 / paths)))
        spp = rng.choice([100, 128, 197, 200, 400])
        periods = max(4, _between(rng, max(1, steps // 16), steps) // spp)
        # at least 2^16 paths: two paths per lane, as the autotuner picks then
        ppt = 2 if paths >= 1 << 16 and what != "normal" else 1
        return {"kind": "run", "what": what, "paths": paths, "spp": spp, "transient": max(1, periods // 10),
                "periods": periods, "block": 64 if ppt == 2 else 128, "ppt": ppt}
    if kind == "scan":
        what = rng.choice(["poisson", "dichot", "both"])
        points = _between(rng, 16, 1024)
        lo = _between(rng, 32, 4096)
        hi = _between(rng, lo, min(16384, 16 * lo))
        periods = max(2, min(300, int(1.5e10 / (points * hi * 100))))
        return {"kind": "scan", "what": what, "points": points, "paths_lo": lo, "paths_hi": hi,
                "spp": rng.choice([100, 200]), "transient": max(1, periods // 10), "periods_lo": max(1, periods // 4),
                "periods_hi": periods, "device": rng.random() < 0.5}
    if kind == "chi":
        return {"kind": "chi", "what": rng.choice(["poisson", "dichot"]), "paths": _between(rng, 512, 16384),
                "spp": rng.choice([100, 200]), "steps": rng.randint(64, 200)}
    if kind == "forward":
        return {"kind": "forward", "rows": _between(rng, 1, 1 << 20)}
    if kind == "screen":
        return {"kind": "screen", "nx": _between(rng, 33, 1024), "ny": _between(rng, 33, 1024)}
    if kind == "fit":
        batch = _between(rng, 64, 4096)
        return {"kind": "fit", "labels": _between(rng, batch, 1 << 17), "batch": batch, "steps": rng.randint(20, 200)}
    return {"kind": "train", "rows": _between(rng, 100, 16384), "steps": rng.randint(1, 4)}


# ---------------------------------------------------------------- inputs

def _params(what, rng):
    """Parameter values of one point: the workloads' with a bias F of the scans'
    range, and the tests' values for the overdamped models."""
    F = float(rng.uniform(-0.3, 0.3))
    if what == "poisson":
        return workloads.poisson_point(F=F)
    if what == "dichot":
        return workloads.dichot_point(F=F)
    if what == "normal":
        return workloads.poisson_point(F=F, noise_flags=GAUSS | POISSON | NORMAL | COMPENSATED)
    both = workloads.poisson_point(F=F, Fa=0.5, Fb=0.5, mua=2.0, mub=2.0, noise_flags=GAUSS | POISSON | DICHOT)
    if what == "both":
        return both
    if what == "washboard":
        return dict(both, V0=0.2, a=0.5, Q=0.05, Fa=0.3, Fb=0.6, mub=1.0)
    return workloads.poisson_point(V0=1.0, a=0.0, F=0.0, Q=0.0, x0_lo=-1.0, x0_hi=1.0, zeta=1.5 / 2.25,
                                   noise_flags=POISSON, **{"lambda": 2.25})


def _model(what):
    return {"washboard": engine.OVERDAMPED_WASHBOARD, "model1": engine.OVERDAMPED_PWL}.get(
        what, engine.INERTIAL_WASHBOARD)


def _dt(case):
    """spp steps per drive period, or per 1 / lambda of Model I."""
    return 1.0 / 2.25 / case["spp"] if case["what"] == "model1" else workloads.period_steps(OMEGA, case["spp"])


def _scan_points(case, seed):
    rng = np.random.default_rng(seed)
    n = case["points"]
    paths = np.exp(rng.uniform(math.log(case["paths_lo"]), math.log(case["paths_hi"] + 1e-9), n)).round().astype(int)
    periods = rng.uniform(case["periods_lo"], case["periods_hi"], n).round().astype(int)
    pts = []
    for i in range(n):
        prm = _params(case["what"], rng)
        if case["what"] == "dichot":
            prm.update(dict.fromkeys(("Fa", "Fb"), float(rng.uniform(0.0, 2.0))))
        else:
            prm.update(Q=float(10.0 ** rng.uniform(-4.0, -1.0)))
        pts.append({"params": engine.make_params(**dict(prm, point=i)), "dt": workloads.period_steps(OMEGA, case["spp"]),
                    "paths": int(paths[i]), "n_transient": case["transient"] * case["spp"],
                    "n_avg": int(periods[i]) * case["spp"]})
    return pts


_SHAPES = [(256, 16), (256,), (256, 256), (256,), (256, 256), (256,), (8, 256), (8,)]
_LIVE = [(256, 7), (256,), (256, 256), (256,), (256, 256), (256,), (2, 256), (2,)]
_LO = [0.5, 2.0, 3.0, -0.3, 1e-4, 0.1, 0.01]
_HI = [1.5, 6.0, 7.0, 0.3, 1e-1, 5.0, 0.5]
_LOG = 1 << 4 | 1 << 5 | 1 << 6


def _weights(seed, off=0.0):
    """Padded parameter vector of a network: Glorot-uniform weights and small
    biases; `off` moves it to a second network that nearly agrees with it."""
    rng, more = np.random.default_rng(seed), np.random.default_rng(seed + 1)
    parts = []
    for shape, live in zip(_SHAPES, _LIVE):
        lim = math.sqrt(6.0 / sum(live)) if len(live) == 2 else 0.05
        w = np.zeros(shape, dtype=np.float32)
        w[tuple(slice(k) for k in live)] = rng.uniform(-lim, lim, live) + off * more.uniform(-lim, lim, live)
        parts.append(w.ravel())
    return np.concatenate(parts)


def _maps():
    """Input map of the seven-parameter box to [-1, 1], output map of (<v>, log10 stderr)."""
    shift, scale = guided.box_maps(_LO, _HI, _LOG)
    return shift, scale, _LOG, [0.05, -3.0], [0.1, 0.5]


def _net(weights):
    net = surrogate.Surrogate(0)
    net.set_maps(*_maps())
    net.set_params(weights)
    return net


def _inputs(rows, seed):
    """Points of the parameter box, log-uniform where the map takes logarithms."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((rows, 7), generator=g, device="cuda", dtype=torch.float64)
    lo, hi = (torch.tensor(v, device="cuda", dtype=torch.float64) for v in (_LO, _HI))
    x = lo + (hi - lo) * u
    x[:, 4:] = torch.exp(torch.log(lo[4:]) + torch.log(hi[4:] / lo[4:]) * u[:, 4:])
    return x.float()


def _labels(x, seed):
    """(<v>, log10 stderr) as a smooth function of the inputs with Monte Carlo noise."""
    g = torch.Generator(device="cuda").manual_seed(seed + 7)
    z = torch.randn((x.shape[0], 2), generator=g, device="cuda")
    v = 0.1 * torch.sin(3.0 * x[:, 3] + x[:, 1]) * torch.cos(x[:, 2]) + 0.05 * x[:, 0] * x[:, 6]
    return torch.stack([v + 1e-3 * z[:, 0], 0.4 * torch.log10(x[:, 4]) - 2.0 + 0.02 * z[:, 1]], 1).contiguous()


def _train_batches(case, seed):
    xs = [_inputs(case["rows"], 100 * seed + k) for k in range(case["steps"])]
    return xs, [_labels(x, 100 * seed + k) for k, x in enumerate(xs)]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("run", "chi"):
        prm = engine.make_params(**_params(case["what"], np.random.default_rng(seed)))
        s["eng"] = engine.Engine(_model(case["what"]), prm, seed=seed)
    if kind == "run":
        s["eng"].set_tuning(case["block"], 0)
        s["eng"].set_paths_per_thread(case["ppt"])
        s["eng"].set_steps_per_launch(case.get("samples", 0))
        n = case["paths"]
        s["out"] = {k: torch.zeros(n, dtype=t, device="cuda") for k, t in (
            ("X_f", torch.float64), ("v_f", torch.float32), ("vbar", torch.float64), ("jP", torch.int32),
            ("jD", torch.int32))}
    elif kind == "scan":
        s["points"] = _scan_points(case, seed)
        s["eng"] = engine.Engine(engine.INERTIAL_WASHBOARD, s["points"][0]["params"], seed=seed)
        s["out5"] = torch.zeros(5 * case["points"], dtype=torch.float64, device="cuda")
    elif kind == "forward":
        s["net"] = _net(_weights(seed))
        s["x"] = _inputs(case["rows"], seed)
    elif kind == "screen":
        s["nets"] = [_net(_weights(seed)), _net(_weights(seed, 0.01))]
        s["x"] = _inputs(case["nx"] * case["ny"], seed)
        s["cal"] = {"kappa": 2.0, "r0": 0.002, "se_scale": 0.5}
    elif kind == "fit":
        s["net"] = _net(_weights(seed))
        s["x"] = _inputs(case["labels"], seed)
        s["t"] = _labels(s["x"], seed)
    elif kind == "train":
        s["net"] = _net(_weights(seed))
        s["x"], s["t"] = _train_batches(case, seed)
        s["loss"] = torch.zeros(case["steps"], device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "run":
        s["eng"].run(case["paths"], _dt(case), case["transient"] * case["spp"], case["periods"] * case["spp"],
                     path_out=s["out"])
        return {"stats": s["eng"].stats(), **s["out"]}
    if kind == "scan":
        if case["device"]:
            s["eng"].scan_device(s["points"], s["out5"])
            return s["out5"]
        res = s["eng"].scan(s["points"])
        return np.array([r["mean_v"] for r in res]), np.array([r["stderr_v"] for r in res]), np.array(
            [r["sums"] for r in res])
    if kind == "chi":
        return s["eng"].local_error(case["paths"], _dt(case), case["steps"])
    if kind == "forward":
        return s["net"].forward(s["x"])
    if kind == "screen":
        v1, v2, lse = guided.predict(s["nets"], s["x"])
        flags, count = guided.select(s["nets"], v1, v2, lse, case["nx"], case["ny"], s["cal"], 0.01, 0.005)
        return {"v1": v1, "v2": v2, "lse": lse, "flags": flags, "count": count}
    if kind == "fit":
        losses = s["net"].fit(s["x"], s["t"], steps=case["steps"], batch=case["batch"], lr=2e-3, lr_final=2e-5, seed=1)
        return {"losses": losses, "params": s["net"].get_params()}
    for k in range(case["steps"]):
        s["net"].train_step(s["x"][k], s["t"][k], 1e-3, loss_out=s["loss"][k:k + 1])
    return {"losses": s["loss"], "params": s["net"].get_params()}


# ---------------------------------------------------------------- what a pass cannot do without

_LIVE_WEIGHTS = 7 * 256 + 2 * 256 * 256 + 2 * 256


def work(case):
    kind = case["kind"]
    if kind in ("run", "scan", "chi"):
        # lane operations of one step of one path: about 40 for the inertial
        # model (force, drive, predictor, corrector, noise), 28 overdamped
        ops = 28.0 if case["what"] in ("model1", "washboard") else 40.0
        if kind == "scan":
            pts = _scan_points(case, 0)
            steps = float(sum(p["paths"] * (p["n_transient"] + p["n_avg"]) for p in pts))
            return {"bytes": 40.0 * case["points"], "flops": ops * steps}
        if kind == "chi":
            return {"bytes": 32.0, "flops": ops * case["paths"] * case["steps"]}
        return {"bytes": 28.0 * case["paths"],
                "flops": ops * case["paths"] * (case["transient"] + case["periods"]) * case["spp"]}
    if kind in ("forward", "screen"):
        rows = case["rows"] if kind == "forward" else 2 * case["nx"] * case["ny"]
        more = 0.0 if kind == "forward" else 13.0 * case["nx"] * case["ny"]
        return {"bytes": 36.0 * rows + more + 4.0 * _LIVE_WEIGHTS, "flops": 2.0 * _LIVE_WEIGHTS * rows}
    rows = case["rows"] if kind == "train" else case["batch"]
    back = 2.0 * (_LIVE_WEIGHTS - 7 * 256)              # no gradient of the inputs
    return {"bytes": case["steps"] * (36.0 * rows + 24.0 * _LIVE_WEIGHTS),
            "flops": case["steps"] * rows * (4.0 * _LIVE_WEIGHTS + back)}


# ---------------------------------------------------------------- values in 64 bits

def _philox(seed, c0, c1, path):
    """Philox4x32-10 words for counters (c0, c1, path, 0); arrays broadcast."""
    m = np.uint64(0xFFFFFFFF)
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    zero = np.zeros(np.broadcast(c0, path).shape, dtype=np.uint64)
    x0, x1 = zero + np.asarray(c0, dtype=np.uint64), zero + np.uint64(c1)
    x2, x3 = zero + np.asarray(path, dtype=np.uint64), zero.copy()
    for _ in range(10):
        p0, p1 = x0 * np.uint64(0xD2511F53), x2 * np.uint64(0xCD9E8D57)
        x0, x1, x2, x3 = (p1 >> np.uint64(32)) ^ x1 ^ k0, p1 & m, (p0 >> np.uint64(32)) ^ x3 ^ k1, p0 & m
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m, (k1 + np.uint64(0xBB67AE85)) & m
    return x0, x1, x2, x3


def _phi(w):
    return (w >> np.uint64(8)).astype(np.float64) / 2.0 ** 24


def _kicks(seed, prm, dt, paths, steps):
    """Poissonian kicks (Algorithm 3): arrays of step, path and amplitude, and
    the number of kicks of each path."""
    p = np.arange(paths)
    at, who, amp = [], [], []
    count = np.zeros(paths, dtype=np.int64)
    step = np.full(paths, -1.0)
    for j in range(steps + 2):
        w = _philox(seed, j >> 1, 2 << 30, p)
        wait, z = (w[0], w[1]) if j % 2 == 0 else (w[2], w[3])
        if j:
            on = step < steps
            at.append(step[on]), who.append(p[on]), amp.append(-prm["zeta"] * np.log(1.0 - _phi(z[on])))
            count += on
        step = step + 1.0 + np.floor(-np.log(1.0 - _phi(wait)) / prm["lambda"] / dt)
        if not (step < steps).any():
            break
    return np.concatenate(at).astype(np.int64), np.concatenate(who), np.concatenate(amp), count


def _flips(seed, prm, dt, paths, steps):
    """Dichotomous state (Algorithm 4) of every step and path."""
    p = np.arange(paths)
    state = _phi(_philox(seed, 0, 0, p)[2]) < prm["mua"] / (prm["mua"] + prm["mub"])
    on = np.zeros((steps, paths), dtype=bool)
    step = np.zeros(paths)
    n = np.arange(steps)[:, None]
    for j in range(steps + 2):
        u = 1.0 - _phi(_philox(seed, j >> 2, 3 << 30, p)[j & 3])
        end = step + (j > 0) + np.floor(-np.log(u) / np.where(state, prm["mub"], prm["mua"]) / dt)
        on |= (n >= step) & (n < end) & state
        state, step = ~state, end
        if not (step < steps).any():
            break
    return on


def _paths64(case, seed, steps, chi):
    """The inertial and the piecewise-linear model in FP64, all paths at once.
    With chi: the local-error indicator; else (X_f, X at the end of the
    transient, kicks per path)."""
    prm = _params(case["what"], np.random.default_rng(seed))
    dt, paths = _dt(case), case["paths"]
    p = np.arange(paths)
    w = _philox(seed, 0, 0, p)
    x = prm["x0_lo"] + (prm["x0_hi"] - prm["x0_lo"]) * _phi(w[0])
    v = prm["v0_lo"] + (prm["v0_hi"] - prm["v0_lo"]) * _phi(w[1])
    flags = prm["noise_flags"]
    count = np.zeros(paths, dtype=np.int64)
    if flags & POISSON:
        at, who, amp, count = _kicks(seed, prm, dt, paths, steps)
        order = np.argsort(at, kind="stable")
        at, who, amp = at[order], who[order], amp[order]
        cut = np.searchsorted(at, np.arange(steps + 1))
    if flags & DICHOT:
        gamma_n = np.where(_flips(seed, prm, dt, paths, steps), prm["Fb"], -prm["Fa"])
    inertial = _model(case["what"]) == engine.INERTIAL_WASHBOARD
    xi = math.sqrt(6.0 * prm["gamma"] * prm["Q"] * dt)
    sums, r, x_i = np.zeros(4), None, x
    two_pi = 2.0 * math.pi
    for n in range(steps):
        jump = np.zeros(paths)
        if flags & POISSON:
            jump -= prm["lambda"] * prm["zeta"] * dt
            jump[who[cut[n]:cut[n + 1]]] += amp[cut[n]:cut[n + 1]]
        if flags & DICHOT:
            jump += gamma_n[n] * dt
        if not inertial:
            force = lambda y: np.where(y - 2.0 * np.floor((y + 1.0) / 2.0) < 0.0, -prm["V0"], prm["V0"]) + prm["F"]
            f1 = force(x)
            pred = x + 0.5 * (f1 + force(x + f1 * dt)) * dt
            x = x + 0.5 * (f1 + force(pred)) * dt + jump
        else:
            d0, d1 = (prm["a"] * math.cos(prm["omega"] * dt * k) + prm["F"] for k in (n, n + 1))
            acc = lambda y, u, d: -prm["gamma"] * u - two_pi * prm["V0"] * np.cos(two_pi * y) + d
            if n % 16 == 0:
                words = _philox(seed, n >> 4, 1 << 30, p)
            r = words[(n >> 2) & 3] if n % 4 == 0 else (r * np.uint64(6)) & np.uint64(0xFFFFFFFF)
            phi = r.astype(np.float64) / 2.0 ** 32
            dxi = np.where(phi <= 1.0 / 6.0, -xi, np.where(phi <= 1.0 / 3.0, xi, 0.0))
            f1 = acc(x, v, d0)
            xb, vb = x + v * dt, v + f1 * dt + dxi
            f2 = acc(xb, vb, d1)
            xp, vp = x + 0.5 * (v + vb) * dt, v + 0.5 * (f1 + f2) * dt + dxi
            f2 = acc(xp, vp, d1)
            x, v = x + 0.5 * (v + vp) * dt, v + 0.5 * (f1 + f2) * dt + dxi
            cx, cv = xp - x, vp - v
            sums += [np.sum(cx * cx), np.sum(cv * cv), 0.0, 0.0]
            sums[2:] = np.maximum(sums[2:], [np.abs(cx).max(), np.abs(cv).max()])
            v = v + jump
        if not chi and n + 1 == case["transient"] * case["spp"]:
            x_i = x
    if chi:
        rms = np.sqrt(sums[:2] / (paths * steps))
        return {"rms_x": float(rms[0]), "rms_v": float(rms[1]), "max_x": float(sums[2]), "max_v": float(sums[3])}
    return x, x_i, count


def _layers64(weights):
    """The layers' weights (rounded to BF16, as the network holds them) and biases."""
    out, at = [], 0
    for k, (shape, live) in enumerate(zip(_SHAPES, _LIVE)):
        n = int(np.prod(shape))
        w = torch.from_numpy(weights[at:at + n].reshape(shape)[tuple(slice(j) for j in live)].copy()).cuda()
        out.append((w.bfloat16() if k % 2 == 0 else w).double())
        at += n
    return out


def _mapped64(x):
    shift, scale, _, _, _ = _maps()
    h = x.double()
    h[:, 4:] = torch.log10(h[:, 4:])
    # the maps are held in FP32
    return (h - torch.from_numpy(np.float32(shift)).cuda().double()) * torch.from_numpy(np.float32(scale)).cuda().double()


def _forward64(weights, x):
    layers = _layers64(weights)
    shift, scale = (torch.tensor(v, dtype=torch.float32).cuda().double() for v in _maps()[3:])
    out = []
    for part in x.split(1 << 17):
        h = _mapped64(part)
        for k in range(4):
            h = torch.nn.functional.linear(h, layers[2 * k], layers[2 * k + 1])
            h = torch.nn.functional.silu(h) if k < 3 else h
        out.append(h * scale + shift)
    return torch.cat(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "chi":
        return _paths64(case, seed, case["steps"], True)
    if kind == "run" and case["what"] == "model1":
        steps = (case["transient"] + case["periods"]) * case["spp"]
        if steps * (case["paths"] + 1000.0) > 1.2e8:                # over about 10 s
            return None
        x, x_i, count = _paths64(case, seed, steps, False)
        vbar = (x - x_i) / (case["periods"] * case["spp"] * _dt(case))
        n = case["paths"]
        stats = dict.fromkeys(("n", "status", "tmean_v", "tvar_v"))
        stats.update(mean_v=float(vbar.mean()), var_v=float(vbar.var(ddof=1)), stderr_v=float(math.sqrt(vbar.var(ddof=1) / n)),
                     sums=[None, float(vbar.sum()), float((vbar ** 2).sum()), None, None])
        return {"stats": stats, "X_f": x, "v_f": None, "vbar": vbar, "jP": None, "jD": None}
    if kind == "forward":
        return _forward64(_weights(seed), _inputs(case["rows"], seed))
    if kind == "screen":
        x = _inputs(case["nx"] * case["ny"], seed)
        y1, y2 = _forward64(_weights(seed), x), _forward64(_weights(seed, 0.01), x)
        return {"v1": y1[:, 0], "v2": y2[:, 0], "lse": 0.5 * (y1[:, 1] + y2[:, 1]), "flags": None, "count": None}
    if kind == "train":
        return _train64(case, seed)
    return None


def _train64(case, seed):
    """The losses of the caller's loop: Adam on FP64 copies, the products on
    BF16-rounded weights."""
    flat = torch.from_numpy(_weights(seed)).cuda().double()
    m1, m2, losses = torch.zeros_like(flat), torch.zeros_like(flat), []
    shift, scale = (torch.tensor(v, dtype=torch.float32).cuda().double() for v in _maps()[3:])
    for k, (x, t) in enumerate(zip(*_train_batches(case, seed))):
        layers = [w.requires_grad_() for w in _layers64(flat.float().cpu().numpy())]
        h = _mapped64(x)
        for j in range(4):
            h = torch.nn.functional.linear(h, layers[2 * j], layers[2 * j + 1])
            h = torch.nn.functional.silu(h) if j < 3 else h
        loss = 0.5 * (h - (t.double() - shift) / scale).square().sum() / x.shape[0]
        losses.append(float(loss.detach()))
        grads, parts = torch.autograd.grad(loss, layers), []
        for g, shape, live in zip(grads, _SHAPES, _LIVE):
            full = torch.zeros(shape, device="cuda", dtype=torch.float64)
            full[tuple(slice(n) for n in live)] = g
            parts.append(full.ravel())
        g = torch.cat(parts)
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        c1, c2 = 1.0 - 0.9 ** (k + 1), 1.0 - 0.999 ** (k + 1)
        flat = flat - 1e-3 * (m1 / c1) / ((m2 / c2).sqrt() + 1e-8)
    return {"losses": torch.tensor(losses, dtype=torch.float64), "params": None}
