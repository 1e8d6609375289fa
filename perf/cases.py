"""Timed cases of the ensemble solver and its surrogate, each a whole pass through the public calls.

A pass is what a program does with new inputs on a context or network that it keeps: hand over the
parameters (``ens_km_coefficients``, ``ens_set_inputs``), solve, wait, read the results into device
arrays; or evaluate, differentiate, train and screen with the surrogate network.  Sizes and settings
follow the workloads of ``paper_2011_01740_gb300.workloads``, the tests and ``bench.py``, with the
horizon of the long sweeps cut to a few forcing periods.  Launch shapes are the library's defaults.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

DEV = "cuda"
PREC = {"fp64": ens.ENS_FP64, "fp32c": ens.ENS_FP32_COMP, "fp32x2": ens.ENS_FP32X2}
WIDTH = 128                       # hidden width of the surrogate network
LAYERS = [(WIDTH, 2), (WIDTH, WIDTH), (WIDTH, WIDTH), (WIDTH, WIDTH), (2, WIDTH)]


# ---------------------------------------------------------------------------
# what is measured
# ---------------------------------------------------------------------------

def listed():
    return [
        # a handful of bubbles, as an interactive exploration or a parameter fit solves them
        dict(name="km_small", kind="km", prec="fp64", pair="ck", dual=False, rows=37, cols=29, phases=2, transient=0),
        # the p_A x f map of 131,044 bubbles at tolerance 1e-10
        dict(name="km_sweep", kind="km", prec="fp64", pair="ck", dual=False, rows=362, cols=362, phases=6,
             transient=0),
        # a frequency-response curve: one amplitude, transient periods first, few systems with long chains
        dict(name="km_frequency", kind="km", prec="fp64", pair="ck", dual=False, rows=1, cols=4608, phases=6,
             transient=4),
        # two driving frequencies with the Dormand-Prince pair
        dict(name="km_dual_dopri5", kind="km", prec="fp64", pair="dp", dual=True, rows=67, cols=91, phases=2,
             transient=0),
        # the map in split precision at tolerance 1e-8
        dict(name="km_split", kind="km", prec="fp32c", pair="ck", dual=False, rows=512, cols=512, phases=4,
             transient=0),
        # the map in double-float arithmetic at tolerance 1e-10
        dict(name="km_doublefloat", kind="km", prec="fp32x2", pair="ck", dual=False, rows=256, cols=256, phases=4,
             transient=0),
        # relief valves with impacts and Poincare points, FP64 and double-float
        dict(name="valve", kind="valve", prec="fp64", n=65536, t1=16.0),
        dict(name="valve_doublefloat", kind="valve", prec="fp32x2", n=131072, t1=16.0),
        # the fixed-step sweep of the Lorenz system
        dict(name="lorenz_rk4", kind="rk4", system="lorenz", n=16384, steps=1000),
        # a trained network screens a parameter grid and hands the doubtful points back
        dict(name="screen", kind="screen", rows=2048, cols=2048, members=4),
        # one gradient of a small, ragged batch (and the predictions on it)
        dict(name="gradient", kind="gradient", n=1000, members=4),
        # training on the solved map, two epochs
        dict(name="train", kind="train", n=130682, batch=8192, epochs=2, members=4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["km", "km", "km", "valve", "valve", "rk4", "screen", "gradient", "train"])
    if kind == "km":
        prec = rng.choice(["fp64", "fp64", "fp64", "fp32c", "fp32x2"])
        pair = rng.choice(["ck", "ck", "dp"]) if prec == "fp64" else "ck"
        rows, cols = rng.choice([1, _log_int(rng, 3, 300)]), _log_int(rng, 5, 400)
        phases = rng.randint(1, 4)
        return dict(kind=kind, prec=prec, pair=pair, dual=rng.random() < 0.25, rows=rows, cols=cols, phases=phases,
                    transient=rng.randint(0, phases - 1))
    if kind == "valve":
        prec = rng.choice(["fp64", "fp32x2"])
        return dict(kind=kind, prec=prec, n=_log_int(rng, 50, 60000 if prec == "fp64" else 120000),
                    t1=float(rng.choice([4, 8, 16])))
    if kind == "rk4":
        return dict(kind=kind, system=rng.choice(["lorenz", "x2p"]), n=_log_int(rng, 100, 262144),
                    steps=_log_int(rng, 50, 2000))
    if kind == "screen":
        return dict(kind=kind, rows=_log_int(rng, 16, 2048), cols=_log_int(rng, 16, 2048), members=rng.randint(2, 4))
    if kind == "gradient":
        return dict(kind=kind, n=_log_int(rng, 64, 16384), members=rng.randint(1, 8))
    return dict(kind=kind, n=_log_int(rng, 2000, 130000), batch=_log_int(rng, 256, 8192), epochs=rng.randint(1, 2),
                members=rng.choice([2, 4]))


# ---------------------------------------------------------------------------
# inputs and kept handles
# ---------------------------------------------------------------------------

class Handle:
    """Owns a context or a network; frees it with the state that holds it."""

    def __init__(self, value, destroy):
        self.value, self._destroy = value, destroy

    def __del__(self):
        self._destroy(self.value)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _km_inputs(case, seed):
    """SI parameters of the map (its corners move a little with the seed) and the initial states."""
    rng = np.random.default_rng(seed)
    pa_max = 2.0e5 * rng.uniform(0.97, 1.0)
    f_min, f_max = 2.0e4 * rng.uniform(1.0, 1.05), 1.0e6 * rng.uniform(0.95, 1.0)
    if case["rows"] == 1:
        w = W.km_frequency_response(case["cols"], pA1=1.5e5 * rng.uniform(0.98, 1.0), f_min=f_min, f_max=f_max)
    else:
        w = W.km(case["rows"], case["cols"], pa_max=pa_max, f_min=f_min, f_max=f_max)
    ph = w["phys"]
    if case["dual"]:
        ph["pA2"], ph["f2"] = 0.5 * ph["pA1"], 2.0 * ph["f1"]
    return {k: _gpu(v) for k, v in ph.items()}, w["liquid"], _gpu(w["y0"])


def _km_tol(case):
    tol = 1e-8 if case["prec"] == "fp32c" else 1e-10
    return ens.make_tol(rtol=tol, atol=tol, dt0=1e-2, dt_min=1e-14, dt_max=1e-1, n_phases=case["phases"],
                        n_transient=case["transient"], prec=PREC[case["prec"]])


def _coefficients(phys, liquid):
    return ens.ens_km_coefficients(*[phys[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], liquid)


def _valve_inputs(case, seed):
    rng = np.random.default_rng(seed)
    w = W.prv(case["n"], q_min=0.2 * rng.uniform(1.0, 1.2), q_max=10.0 * rng.uniform(0.98, 1.0), t1=case["t1"])
    return _gpu(w["params"]), _gpu(w["y0"]), w["tol"]


def _rk4_inputs(case, seed):
    rng = np.random.default_rng(seed)
    if case["system"] == "lorenz":
        w = W.lorenz(case["n"], rho_max=21.0 * rng.uniform(0.95, 1.0))
        w["y0"] = w["y0"] * rng.uniform(0.99, 1.01)
    else:
        w = W.x2p(case["n"])
        w["params"] = w["params"] * rng.uniform(0.95, 1.0)
    return _gpu(w["params"]), _gpu(w["y0"]), w["dt"]


def _samples(n, seed):
    """Feature points in [-1, 1]^2 with a smooth response and a 0 / 1 label."""
    x, y = W.mlp_batch(n, seed=seed)
    return _gpu(x), _gpu(y)


def _network(case, seed, gain=1.0):
    p = _gpu(np.float32(gain) * W.mlp_params(case["members"], seed=seed))
    m = Handle(ens.ens_mlp_create(case["members"], seed), ens.ens_mlp_destroy)
    ens.ens_mlp_set_params(m.value, p)
    return m, p


def _outputs(ctx, rows):
    n, d = ens.ens_size(ctx), ens.ens_dim(ctx)
    out = dict(state=torch.empty((d, n), dtype=torch.float64, device=DEV),
               status=torch.empty(n, dtype=torch.int32, device=DEV),
               steps=torch.empty(n, dtype=torch.int64, device=DEV))
    if rows:
        out["acc"] = torch.empty((rows, n), dtype=torch.float64, device=DEV)
    return out


def prepare(case, seed):
    s = dict(case=case)
    if case["kind"] == "km":
        phys, liquid, y0 = _km_inputs(case, seed)
        solver = ens.ENS_DOPRI5 if case["pair"] == "dp" else ens.ENS_RKCK45
        ctx = ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, y0.shape[1], _coefficients(phys, liquid), y0, (0.0, 1.0),
                             solver, _km_tol(case))
        s.update(phys=phys, liquid=liquid, y0=y0)
    elif case["kind"] == "valve":
        params, y0, t = _valve_inputs(case, seed)
        tol = ens.make_tol(rtol=t.rtol, atol=t.atol, dt0=t.dt0, dt_min=t.dt_min, dt_max=t.dt_max,
                           event_tol=t.event_tol, acc_t_start=t.acc_t_start, prec=PREC[case["prec"]])
        ctx = ens.ens_create(ens.ENS_SYS_RELIEF_VALVE, case["n"], params, y0, (t.t0, t.t1), ens.ENS_RKCK45, tol)
        s.update(params=params, y0=y0)
    elif case["kind"] == "rk4":
        params, y0, dt = _rk4_inputs(case, seed)
        system = ens.ENS_SYS_LORENZ if case["system"] == "lorenz" else ens.ENS_SYS_TOY_X2P
        ctx = ens.ens_create(system, case["n"], params, y0, (0.0, dt * case["steps"]), ens.ENS_RK4,
                             ens.make_tol(dt0=dt, n_steps=case["steps"]))
        s.update(params=params, y0=y0)
    elif case["kind"] == "screen":
        rng = np.random.default_rng(seed)
        pa = W.logspace(2.0e5 / 361, 2.0e5 * rng.uniform(0.9, 1.0), case["rows"])
        f = W.logspace(2.0e4, 1.0e6 * rng.uniform(0.9, 1.0), case["cols"])
        PA, F = np.meshgrid(pa, f, indexing="ij")
        n = pa.size * f.size
        s["net"], s["weights"] = _network(case, seed, gain=1.5)   # a response as steep as a trained network's
        s.update(pa=_gpu(PA.ravel()), f=_gpu(F.ravel()), x=torch.empty((n, 2), dtype=torch.float32, device=DEV),
                 idx=torch.full((n,), -1, dtype=torch.int32, device=DEV),
                 **{k: torch.zeros(n, dtype=torch.float64, device=DEV) for k in ("pa_back", "f_back")},
                 **{k: torch.empty(n, dtype=torch.float32, device=DEV) for k in ("mean", "stdv", "p1", "slope")})
        return s
    else:
        s["x"], s["y"] = _samples(case["n"], seed)
        s["net"], s["weights"] = _network(case, seed)
        s["grad"] = torch.empty_like(s["weights"])
        s["out"] = torch.empty((case["members"], case["n"], 2), dtype=torch.float32, device=DEV)
        s["cfg"] = _train_cfg(case, seed) if case["kind"] == "train" else None
        return s
    s["ctx"] = Handle(ctx, ens.ens_destroy)
    s["read"] = _outputs(ctx, ens.ens_acc_rows(ctx))
    return s


def _train_cfg(case, seed):
    return ens.make_train_cfg(epochs=case["epochs"], batch=case["batch"], lr=2e-3, seed=seed, lr_final=2e-5)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

SELECT = dict(state=ens.ENS_STATE, acc=ens.ENS_ACC, status=ens.ENS_STATUS, steps=ens.ENS_NSTEPS)
SPREAD, SLOPE = 0.85, 1.2         # fallback gates of the screen: ensemble spread, steepness


def run(s):
    case = s["case"]
    if case["kind"] == "screen":
        return _screen(s)
    if case["kind"] == "gradient":
        m = s["net"].value
        ens.ens_mlp_forward(m, case["n"], s["x"], s["out"])
        loss = ens.ens_mlp_loss_grad(m, case["n"], s["x"], s["y"], case["members"], s["grad"])
        return dict(out=s["out"], loss=loss, grad=s["grad"])
    if case["kind"] == "train":
        m = s["net"].value
        ens.ens_mlp_set_params(m, s["weights"])          # from the given weights, Adam moments at zero
        loss = ens.ens_mlp_train(m, case["n"], s["x"], s["y"], s["cfg"], case["members"])
        return dict(loss=loss, weights=ens.ens_mlp_get_params(m, s["grad"]))
    ctx = s["ctx"].value
    params = _coefficients(s["phys"], s["liquid"]) if case["kind"] == "km" else s["params"]
    ens.ens_set_inputs(ctx, params, s["y0"])
    ens.ens_solve(ctx)
    ens.ens_sync(ctx)
    for k, dst in s["read"].items():
        ens.ens_read(ctx, SELECT[k], dst)
    return s["read"]


def _spacings(case):
    return 2.0 / max(1, case["rows"] - 1), 2.0 / max(1, case["cols"] - 1)


def _stride(case):
    return max(1, min(case["rows"], case["cols"]) // 16)


def _screen(s):
    case, m, n = s["case"], s["net"].value, s["x"].shape[0]
    dr, dc = _spacings(case)
    ens.ens_km_features(n, s["pa"], s["f"], W.KM_FEATURE_RANGE, s["x"])
    ens.ens_mlp_screen(m, n, s["x"], s["mean"], s["stdv"], s["p1"])
    ens.ens_grid_gradient(case["rows"], case["cols"], _stride(case), s["mean"], dr, dc, s["slope"])
    k = ens.ens_select_gate(n, s["stdv"], SPREAD, s["slope"], SLOPE, s["idx"])
    ens.ens_gather_f64(k, s["idx"], s["pa"], s["pa_back"])     # the flagged points, for the solver
    ens.ens_gather_f64(k, s["idx"], s["f"], s["f_back"])
    return dict({key: s[key] for key in ("mean", "stdv", "p1", "slope", "idx", "pa_back", "f_back")}, count=k)


# ---------------------------------------------------------------------------
# the least work of a pass
# ---------------------------------------------------------------------------

def _trials(case):
    """About how many trial steps a system takes: 560 per period at 1e-10 on the map, in proportion to
    tol^(-1/5) for the fifth-order pairs; 126 per time unit for the valve."""
    if case["kind"] == "valve":
        return 126.0 * case["t1"]
    return 560.0 * case["phases"] * (100.0 ** -0.2 if case["prec"] == "fp32c" else 1.0)


def work(case):
    if case["kind"] == "km":
        n = case["rows"] * case["cols"]
        per_trial = 590.0 * (1.2 if case["pair"] == "dp" else 1.0) * (1.4 if case["dual"] else 1.0)
        rows = 2 * (case["phases"] - case["transient"])
        return dict(bytes=n * (8.0 * (6 + 2 + 2 + rows) + 12), flops=n * _trials(case) * per_trial)
    if case["kind"] == "valve":
        n = case["n"]
        return dict(bytes=n * (8.0 * (5 + 3 + 3 + 35) + 12), flops=n * _trials(case) * 302.0)
    if case["kind"] == "rk4":
        d, p, flops = (3, 3, 75.0) if case["system"] == "lorenz" else (1, 1, 21.0)
        return dict(bytes=case["n"] * (8.0 * (p + 2 * d) + 12), flops=case["n"] * case["steps"] * flops)
    macs = sum(a * b for a, b in LAYERS)
    floats = sum(a * b + a for a, b in LAYERS) * case["members"]
    if case["kind"] == "screen":
        n = case["rows"] * case["cols"]
        return dict(bytes=n * 32.0 + floats * 4.0, flops=2.0 * macs * case["members"] * n)
    if case["kind"] == "gradient":
        return dict(bytes=case["n"] * 8.0 * (2 + case["members"]) + floats * 8.0,
                    flops=8.0 * macs * case["members"] * case["n"])
    return dict(bytes=case["epochs"] * case["n"] * 16.0 + floats * 8.0,
                flops=6.0 * macs * case["members"] * case["n"] * case["epochs"])


# ---------------------------------------------------------------------------
# the same results from plain 64-bit arithmetic
# ---------------------------------------------------------------------------

def exact(case, seed):
    if case["kind"] == "km":
        # a lock-step loop over the longest system's steps: minutes for the larger maps
        return _exact_km(case, seed) if case["phases"] <= 2 and case["rows"] * case["cols"] <= 20000 else None
    if case["kind"] == "valve":
        return _exact_valve(case, seed) if case["t1"] <= 8 and case["n"] <= 20000 else None
    if case["kind"] == "rk4":
        return _exact_rk4(case, seed)
    if case["kind"] == "screen":
        return _exact_screen(case, seed)
    if case["kind"] == "gradient":
        x, y = (t.double() for t in _samples(case["n"], seed))
        p = _gpu(W.mlp_params(case["members"], seed=seed)).double()
        out, loss, grad = _loss_grad64(p, x, y)
        return dict(out=out, loss=loss, grad=grad)
    return _exact_train(case, seed)


CK = ([[1 / 5], [3 / 40, 9 / 40], [3 / 10, -9 / 10, 6 / 5], [-11 / 54, 5 / 2, -70 / 27, 35 / 27],
       [1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096]],
      [1 / 5, 3 / 10, 3 / 5, 1.0, 7 / 8], [37 / 378, 0.0, 250 / 621, 125 / 594, 0.0, 512 / 1771],
      [2825 / 27648, 0.0, 18575 / 48384, 13525 / 55296, 277 / 14336, 1 / 4])
DP = ([[1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9], [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
       [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
       [35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]],
      [1 / 5, 3 / 10, 4 / 5, 8 / 9, 1.0, 1.0], [35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0.0],
      [5179 / 57600, 0.0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40])


def _trial64(f, pair, t, h, y, tol):
    """One embedded Runge-Kutta trial: the first slope, the fifth-order state, the error norm, the step factor."""
    a, c, b, bs = pair
    k = [f(t, y)]
    for row, ci in zip(a, c):
        k.append(f(t + ci * h, y + h * sum(w * ki for w, ki in zip(row, k) if w)))
    new = y + h * sum(w * ki for w, ki in zip(b, k) if w)
    err = h * sum((w - ws) * ki for w, ws, ki in zip(b, bs, k) if w != ws)
    e = (err.abs() / (tol + tol * torch.maximum(y.abs(), new.abs()))).amax(0)
    fac = (0.9 * e.clamp(1e-4, 2000.0) ** -0.2).clamp(0.2, 5.0)
    return k[0], new, e, torch.where(e.isnan(), torch.full_like(fac, 0.2), fac)


def _km_rhs(C):
    tp = 2.0 * math.pi

    def f(t, y):
        y1, y2 = y[0], y[1]
        fs, fc = C[5] * torch.sin(tp * t), C[7] * torch.cos(tp * t)
        fs = fs + C[6] * torch.sin(tp * C[11] * t + C[12])
        fc = fc + C[8] * torch.cos(tp * C[11] * t + C[12])
        m = 1.0 + C[9] * y2
        N = (C[0] + C[1] * y2) * y1 ** -C[10] - C[2] * m - (C[3] + C[4] * y2) / y1
        N = N - (1.5 - 0.5 * C[9] * y2) * y2 * y2 - fs * m - y1 * fc
        return torch.stack([y2, N / (y1 * (1.0 - C[9] * y2) + C[4] * C[9])])
    return f


def _km_coefficients64(ph, L):
    """C0..C12 from the SI parameters (the paper's coefficient equations)."""
    w1, w2 = 2 * math.pi * ph["f1"], 2 * math.pi * ph["f2"]
    s = 2 * math.pi / (ph["RE"] * w1)
    pg = L["pinf"] - L["pv"] + 2 * L["sigma"] / ph["RE"]
    rc, one = L["rho"] * L["c"], torch.ones_like(w1)
    return torch.stack([pg / L["rho"] * s**2, (1 - 3 * L["gamma"]) / rc * pg * s, (L["pinf"] - L["pv"]) / L["rho"] * s**2,
                        2 * L["sigma"] / (L["rho"] * ph["RE"]) * s**2,
                        4 * L["mu"] / (L["rho"] * ph["RE"]**2) * 2 * math.pi / w1, ph["pA1"] / L["rho"] * s**2,
                        ph["pA2"] / L["rho"] * s**2, ph["RE"] * w1 * ph["pA1"] / rc * s**2,
                        ph["RE"] * w2 * ph["pA2"] / rc * s**2, ph["RE"] * w1 / (2 * math.pi * L["c"]),
                        3 * L["gamma"] * one, w2 / w1, ph["theta"]])


def _exact_km(case, seed):
    """Phase-mode integration of all systems in lock step; finished ones are dropped every 64 trials."""
    phys, liquid, y0 = _km_inputs(case, seed)
    C, n, tol = _km_coefficients64(phys, liquid), y0.shape[1], _km_tol(case).rtol
    rec = case["phases"] - case["transient"]
    acc = torch.full((2 * rec, n), float("nan"), dtype=torch.float64, device=DEV)
    state = y0.clone()
    ids, y = torch.arange(n, device=DEV), y0.clone()
    t, dt, ph = (torch.full((n,), v, dtype=torch.float64, device=DEV) for v in (0.0, 1e-2, 0.0))
    hi, lo, pair = y[0].clone(), y[0].clone(), (DP if case["pair"] == "dp" else CK)
    it, f = 0, _km_rhs(C)
    while ids.numel():
        live = ph < case["phases"]
        clamped = dt >= 1.0 - t
        h = torch.where(clamped, 1.0 - t, dt)
        _, new, e, fac = _trial64(f, pair, t, h, y, tol)
        ok = (e <= 1.0) & live
        y = torch.where(ok, new, y)
        t = torch.where(ok, torch.where(clamped, torch.ones_like(t), t + h), t)
        dt = torch.where(ok & clamped, dt, torch.where(live, (h * fac).clamp(1e-14, 1e-1), dt))
        hi, lo = torch.where(ok, torch.maximum(hi, y[0]), hi), torch.where(ok, torch.minimum(lo, y[0]), lo)
        end = ok & (t >= 1.0)
        put = end & (ph >= case["transient"])
        r = torch.where(put, ph - case["transient"], torch.zeros_like(ph)).long()
        for k, v in ((0, hi), (1, lo)):
            acc[2 * r + k, ids] = torch.where(put, v, acc[2 * r + k, ids])
        ph = ph + end
        t = torch.where(end & (ph < case["phases"]), torch.zeros_like(t), t)
        hi, lo = torch.where(end, y[0], hi), torch.where(end, y[0], lo)
        it += 1
        if it % 64 == 0:
            state[:, ids] = y
            keep = ph < case["phases"]
            ids, y, t, dt, ph, hi, lo, C = (v[..., keep] for v in (ids, y, t, dt, ph, hi, lo, C))
            f = _km_rhs(C)
    return dict(state=state, acc=acc, status=None, steps=None)


def _event_root(g, dg, g1, h):
    """The fraction of h at which the parabola through g with slope dg and through g1 at h vanishes."""
    B = h * dg
    A = g1 - g - B
    x = 2 * g / (torch.sqrt((B * B - 4 * A * g).clamp(min=0)) - B)
    return torch.where((x > 0) & (x < 1), x, g / (g - g1))


def _exact_valve(case, seed):
    """Event-mode integration of all valves in lock step (impacts, Poincare points, rest on the seat)."""
    params, y, tl = _valve_inputs(case, seed)
    q, kappa, delta, beta, r = params
    n, t1, tol, band = case["n"], tl.t1, tl.rtol, tl.event_tol

    def f(_, y):
        return torch.stack([y[1], -kappa * y[1] - (y[0] + delta) + y[2],
                            beta * (q - y[0] * torch.sqrt(y[2].clamp(min=0)))])

    zero = torch.zeros(n, dtype=torch.float64, device=DEV)
    t, dt, hev, ymin = zero.clone(), zero + tl.dt0, zero.clone(), zero + math.inf
    nmax, nimp = zero.clone(), zero.clone()
    ring = torch.full((32, n), float("nan"), dtype=torch.float64, device=DEV)
    ids, stuck = torch.arange(n, device=DEV), zero > 1
    while bool((t < t1).any()):
        for _ in range(16):
            live = (t < t1) & ~stuck
            lift = t + (delta - y[2]) / (beta * q)
            sit = (t < t1) & stuck
            y3 = torch.where(lift >= t1, y[2] + beta * q * (t1 - t), delta)
            stuck = stuck & ~(sit & (lift < t1))
            t_sit = torch.minimum(lift, zero + t1)
            last = dt >= t1 - t
            h = torch.where(last, t1 - t, dt)
            cut = (hev > 0) & (hev < h)
            h = torch.where(cut, hev, h)
            k1, new, e, fac = _trial64(f, CK, t, h, y, tol)
            good = (e <= 1.0) & live
            o1 = good & (new[0] < -band)
            o2 = good & (y[1] > band) & (new[1] < -band)
            x1 = torch.where(y[0] > band, _event_root(y[0], k1[0], new[0], h), zero + 0.5)
            x2 = _event_root(y[1], k1[1], new[1], h)
            best = torch.minimum(torch.where(o1, x1, zero + 2), torch.where(o2, x2, zero + 2))
            over = o1 | o2
            ok = good & ~over
            old = y[1]
            y = torch.where(ok, new, y)
            t = torch.where(ok, torch.where(last & ~cut, zero + t1, t + h), torch.where(sit, t_sit, t))
            dt = torch.where(ok & ~last & ~cut, (h * fac).clamp(tl.dt_min, tl.dt_max),
                             torch.where(live & ~good, h * fac, dt))
            hev = torch.where(over, h * best, torch.where(live, zero, hev))
            top = ok & (old > band) & (y[1].abs() <= band)
            slot = (nmax % 32).long()
            ring[slot, ids] = torch.where(top, y[0], ring[slot, ids])
            nmax = nmax + top
            hit = ok & (y[0].abs() <= band) & (y[1] < 0)
            push = delta - y[2]
            v = torch.where(hit, -r * y[1], y[1])
            rest = hit & (push > 0) & (v * v <= 2 * push * band)
            y = torch.stack([torch.where(hit, zero, y[0]), torch.where(rest, zero, v), torch.where(sit, y3, y[2])])
            nimp, stuck = nimp + hit, stuck | rest
            ymin = torch.where((ok | sit) & (t >= tl.acc_t_start), torch.minimum(ymin, y[0]), ymin)
    return dict(state=y, acc=torch.cat([ring, torch.stack([ymin, nmax, nimp])]), status=None, steps=None)


def _exact_rk4(case, seed):
    p, y, h = _rk4_inputs(case, seed)
    if case["system"] == "lorenz":
        def f(y):
            return torch.stack([p[1] * (y[1] - y[0]), p[0] * y[0] - y[1] - y[0] * y[2], y[0] * y[1] - p[2] * y[2]])
    else:
        def f(y):
            return y * y - p
    for _ in range(case["steps"]):
        k1 = f(y)
        k2 = f(y + 0.5 * h * k1)
        k3 = f(y + 0.5 * h * k2)
        k4 = f(y + h * k3)
        y = y + h / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
    return dict(state=y, status=None, steps=None)


def _parts(p):
    """Weights and biases of the members' parameter vectors p [members][count]."""
    at, got = 0, []
    for a, b in LAYERS:
        got.append((p[:, at:at + a * b].reshape(-1, a, b), p[:, at + a * b:at + a * b + a]))
        at += a * b + a
    return got


def _forward64(p, x):
    h = x.expand(p.shape[0], -1, -1)
    for k, (w, b) in enumerate(_parts(p)):
        h = torch.baddbmm(b[:, None, :], h, w.transpose(1, 2))
        if k < 4:
            h = torch.nn.functional.gelu(h)
    return h


def _loss_grad64(p, x, y):
    """Outputs, mean loss and its gradient for every member."""
    p = p.detach().requires_grad_(True)
    out = _forward64(p, x)
    loss = ((out[..., 0] - y[:, 0]) ** 2).mean(1) + torch.nn.functional.binary_cross_entropy_with_logits(
        out[..., 1], y[:, 1].expand(p.shape[0], -1), reduction="none").mean(1)
    grad, = torch.autograd.grad(loss.sum(), p)
    return out.detach(), loss.detach(), grad


def _exact_screen(case, seed):
    s = prepare(case, seed)
    lo, hi, flo, fhi = W.KM_FEATURE_RANGE
    x = torch.stack([2 * (torch.log(s["pa"]) - math.log(lo)) / (math.log(hi) - math.log(lo)) - 1,
                     2 * (torch.log(s["f"]) - math.log(flo)) / (math.log(fhi) - math.log(flo)) - 1], 1)
    p = s["weights"].double()
    out = torch.cat([_forward64(p, c) for c in x.split(1 << 17)], 1)
    mean, stdv, p1 = out[..., 0].mean(0), out[..., 0].std(0, unbiased=False), torch.sigmoid(out[..., 1]).mean(0)
    g, st, (dr, dc) = mean.reshape(case["rows"], case["cols"]), _stride(case), _spacings(case)
    slope = torch.zeros_like(g)
    if st < case["rows"]:
        d = (g[st:] - g[:-st]).abs() / (dr * st)
        slope[st:], slope[:-st] = torch.maximum(slope[st:], d), torch.maximum(slope[:-st], d)
    if st < case["cols"]:
        d = (g[:, st:] - g[:, :-st]).abs() / (dc * st)
        slope[:, st:], slope[:, :-st] = torch.maximum(slope[:, st:], d), torch.maximum(slope[:, :-st], d)
    return dict(mean=mean, stdv=stdv, p1=p1, slope=slope.reshape(-1), idx=None, pa_back=None, f_back=None,
                count=None)


def _splitmix64(c):
    """Draws of the shuffle's counter-based generator for the counters c (uint64)."""
    x = c + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def _shuffle(n, seed, epoch):
    start = np.uint64((seed + 0x51ED2701 * (epoch + 1)) % 2**44 * 2**20)
    i = np.arange(n - 1, 0, -1, dtype=np.uint64)
    at = _splitmix64(start + np.arange(n - 1, dtype=np.uint64)) % (i + np.uint64(1))
    p = list(range(n))
    for a, b in zip(i.tolist(), at.tolist()):
        p[a], p[b] = p[b], p[a]
    return torch.tensor(p, device=DEV)


def _exact_train(case, seed):
    n, B, cfg = case["n"], min(case["batch"], case["n"]), _train_cfg(case, seed)
    x, y = (t.double() for t in _samples(n, seed))
    p = _gpu(W.mlp_params(case["members"], seed=seed)).double()
    m1, m2, hist, step = torch.zeros_like(p), torch.zeros_like(p), [], 0
    total = case["epochs"] * (-(-n // B))
    for ep in range(case["epochs"]):
        perm, lsum = _shuffle(n, seed, ep), 0.0
        for at in perm.split(B):
            _, loss, g = _loss_grad64(p, x[at], y[at])
            lsum = lsum + loss * at.numel()
            lr = cfg.lr_final + 0.5 * (cfg.lr - cfg.lr_final) * (1 + math.cos(math.pi * step / (total - 1))) \
                if total > 1 else cfg.lr
            step += 1
            m1, m2 = cfg.beta1 * m1 + (1 - cfg.beta1) * g, cfg.beta2 * m2 + (1 - cfg.beta2) * g * g
            p = p - lr * (m1 / (1 - cfg.beta1**step)) / ((m2 / (1 - cfg.beta2**step)).sqrt() + cfg.eps)
        hist.append(lsum / n)
    return dict(loss=torch.stack(hist), weights=p)
