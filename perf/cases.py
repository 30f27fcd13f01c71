"""Performance cases: calls that programs built on this package make.

Implied volatilities of a smile and of a whole book, calibrations by Simulated
Annealing (one smile, a surface of smiles, joint dynamic fits, both
precisions), Monte Carlo prices (log-Euler, conditional-Bessel, cliquet) and a
burst of calibration requests to the server.  Every call goes through the
package's public entry points; inputs are formed here, from the seed alone, by
plain NumPy in 64 bits.

A case is a dict of plain values with a "kind"; listed() gives the named ones,
draw(rng) another of the same ranges.
"""
import math

import numpy as np
import torch

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

MODELS = {"hagan": sg.HAGAN, "obloj": sg.OBLOJ, "expanded": sg.EXPANDED, "dyn1": sg.DYN_I, "dyn2": sg.DYN_II}
PRECS = {"fp32": sg.FP32, "fp64": sg.FP64}
BOXES = {"hagan": (W.STATIC_LO, W.STATIC_HI), "obloj": (W.STATIC_LO, W.STATIC_HI),
         "expanded": (W.STATIC_LO, W.STATIC_HI), "dyn1": (W.DYN1_LO, W.DYN1_HI), "dyn2": (W.DYN2_LO, W.DYN2_HI)}


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one smile's volatilities: the smallest call, as in re-marking a quote screen
        {"name": "vol_smile", "kind": "vol", "model": "hagan", "prec": "fp32", "n": 21},
        # a whole option book marked at once (the test suite's large launch, made ragged)
        {"name": "vol_book", "kind": "vol", "model": "hagan", "prec": "fp32", "n": (1 << 20) - 3},
        # one 15-strike smile, 64 chains, 200 x 100: the smallest calibration
        {"name": "smile", "kind": "calibrate", "model": "hagan", "prec": "fp32", "mats": 1, "strikes": 15,
         "chains": 64, "levels": 200, "len": 100},
        # the same smile in the FP64 form, as a check of a production fit
        {"name": "smile_fp64", "kind": "calibrate", "model": "hagan", "prec": "fp64", "mats": 1, "strikes": 15,
         "chains": 64, "levels": 200, "len": 100},
        # the benchmark's static surface: ten 21-strike smiles, 4096 chains each, one resident plan
        {"name": "surface", "kind": "surface", "model": "hagan", "prec": "fp32", "smiles": 10, "strikes": 21,
         "chains": 4096, "levels": 200, "len": 100},
        # the joint dynamic fits of 12 maturities x 21 strikes (Cases I and II), the largest calibrations
        {"name": "dynamic1", "kind": "calibrate", "model": "dyn1", "prec": "fp32", "mats": 12, "strikes": 21,
         "chains": 8192, "levels": 200, "len": 100},
        {"name": "dynamic2", "kind": "calibrate", "model": "dyn2", "prec": "fp32", "mats": 12, "strikes": 21,
         "chains": 8192, "levels": 200, "len": 100},
        # a call surface priced with the paths of one calibration evaluation
        {"name": "mc_small", "kind": "mc", "model": "hagan", "prec": "fp32", "scheme": "euler", "mats": 8,
         "strikes": 15, "paths": 1 << 16, "spy": 250},
        # the same surface at pricing accuracy, the largest pricing call
        {"name": "mc_large", "kind": "mc", "model": "hagan", "prec": "fp32", "scheme": "euler", "mats": 8,
         "strikes": 15, "paths": 1 << 22, "spy": 250},
        # the low-bias scheme on its coarse grid
        {"name": "mc_bessel", "kind": "mc", "model": "hagan", "prec": "fp32", "scheme": "bessel", "mats": 8,
         "strikes": 15, "paths": (1 << 20) + 77, "spy": 12},
        # the paper's exotic: a quarterly cliquet on the dynamic model
        {"name": "cliquet", "kind": "cliquet", "model": "dyn1", "prec": "fp32", "resets": 4, "paths": 1 << 20,
         "spy": 250},
        # a burst of requests of uneven size to the server, one of them calibrated to Monte Carlo prices
        {"name": "serving", "kind": "serving", "requests": 20, "mc_requests": 1, "chains": 1024, "levels": 100,
         "len": 50, "mc_paths": 1 << 14},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vol", "vol", "calibrate", "calibrate", "surface", "joint", "mc", "mc", "bessel", "cliquet",
                       "serving"])
    if kind == "vol":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        model = rng.choice(list(MODELS))
        top = 1 << 20 if prec == "fp32" else (1 << 12 if model == "dyn2" else 1 << 17)
        return {"kind": "vol", "model": model, "prec": prec, "n": _log_int(rng, 1, top)}
    if kind == "calibrate":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        wide = prec == "fp32"
        return {"kind": "calibrate", "model": rng.choice(["hagan", "hagan", "obloj", "expanded"]), "prec": prec,
                "mats": rng.randint(1, 12 if wide else 2), "strikes": rng.randint(5, 41 if wide else 21),
                "chains": _log_int(rng, 48, 2048 if wide else 64), "levels": rng.randint(20, 100),
                "len": rng.randint(20, 100)}
    if kind == "surface":
        return {"kind": "surface", "model": "hagan", "prec": "fp32", "smiles": rng.randint(2, 10),
                "strikes": rng.randint(5, 41), "chains": _log_int(rng, 200, 4096), "levels": rng.randint(20, 100),
                "len": rng.randint(20, 100)}
    if kind == "joint":
        return {"kind": "calibrate", "model": rng.choice(["dyn1", "dyn2"]), "prec": "fp32",
                "mats": rng.randint(1, 12), "strikes": rng.randint(5, 41), "chains": _log_int(rng, 200, 8192),
                "levels": rng.randint(10, 60), "len": rng.randint(20, 100)}
    if kind == "mc":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        return {"kind": "mc", "model": rng.choice(["hagan", "dyn1", "dyn2"]), "prec": prec, "scheme": "euler",
                "mats": rng.randint(1, 8), "strikes": rng.randint(1, 21),
                "paths": _log_int(rng, 1000, 1 << 21 if prec == "fp32" else 1 << 15),
                "spy": rng.choice([12, 50, 100, 250])}
    if kind == "bessel":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        return {"kind": "mc", "model": rng.choice(["hagan", "dyn1", "dyn2"]), "prec": prec, "scheme": "bessel",
                "mats": rng.randint(1, 8), "strikes": rng.randint(1, 21),
                "paths": _log_int(rng, 1000, 1 << 20 if prec == "fp32" else 1 << 15), "spy": rng.choice([4, 12, 16])}
    if kind == "cliquet":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        return {"kind": "cliquet", "model": rng.choice(["hagan", "dyn1", "dyn2"]), "prec": prec,
                "resets": rng.choice([3, 4, 6, 12]),
                "paths": _log_int(rng, 1000, 1 << 20 if prec == "fp32" else 1 << 15),
                "spy": rng.choice([12, 50, 100, 250])}
    return {"kind": "serving", "requests": rng.randint(3, 20), "mc_requests": rng.randint(0, 1),
            "chains": _log_int(rng, 256, 1024), "levels": rng.randint(20, 100), "len": rng.randint(20, 50),
            "mc_paths": _log_int(rng, 4096, 1 << 14)}


# ---------------------------------------------------------------------------
# The volatility formulas in 64-bit NumPy: they form the markets that the
# calibrations are given, and say what a volatility call should return
# ---------------------------------------------------------------------------
def _z_over_x(z, rho):
    D = np.sqrt((z - rho) ** 2 + (1 - rho) * (1 + rho))
    with np.errstate(all="ignore"):
        x = np.where(z > 1, np.log1p((D + z - 1) / (1 - rho)),
                     np.where(z < -1, np.log((1 + rho) / (D - z + rho)), np.log1p(2 * z / (1 - z + D))))
        return np.where(z == 0, 1.0, z / x)


def _panels(T, k):
    """A composite 20-point Gauss-Legendre rule on [0, T] that resolves rates up to k / T."""
    x, w = np.polynomial.legendre.leggauss(20)
    n = 1 + int(math.ceil(k / 4))
    e = np.linspace(0.0, T, n + 1)
    h = 0.5 * np.diff(e)[:, None]
    return ((e[:-1, None] + h) + h * x).ravel(), (h * w).ravel()


def _term_functions(p, T):
    """nu1^2, nu2^2, eta1 and eta2^2 at maturity T (Sec. 2.2), by quadrature."""
    a, b = p[4], p[5]
    nu = lambda t: (p[3] + p[9] * t) * np.exp(-b * t) + p[7]
    rho = lambda t: (p[2] + p[8] * t) * np.exp(-a * t) + p[6]
    k = max(2 * b, a + b) * T
    t, w = _panels(T, k)
    u, v = _panels(1.0, k)
    s = t[:, None] * u
    G = t * ((nu(s) * rho(s)) @ v)
    return (3 / T ** 3 * np.sum(w * (T - t) ** 2 * nu(t) ** 2), 6 / T ** 3 * np.sum(w * (T - t) * t * nu(t) ** 2),
            2 / T ** 2 * np.sum(w * (T - t) * nu(t) * rho(t)), 12 / T ** 4 * np.sum(w * (T - t) * G ** 2))


def _vols(model, p, f, T, K):
    """Implied volatilities of a model, 64-bit."""
    T, K = np.asarray(T, dtype=np.float64), np.asarray(K, dtype=np.float64)
    p = np.concatenate([np.asarray(p, dtype=np.float64), np.zeros(10)])[:10]
    al, be, rho, nu = p[:4]
    L, o = np.log(f / K), 1 - be
    if model in ("hagan", "obloj"):
        fk = (f * K) ** (o / 2)
        z = nu / al * (L * fk if model == "hagan" else
                       (K ** o * np.expm1(o * L) / o if o != 0 else L))
        den = 1 + o ** 2 / 24 * L ** 2 + o ** 4 / 1920 * L ** 4
        br = 1 + (o ** 2 / 24 * al ** 2 / fk ** 2 + rho * be * nu * al / (4 * fk) + (2 - 3 * rho ** 2) / 24 * nu ** 2) * T
        if model == "hagan":
            lead = al / fk
        else:
            zd = K ** o * np.expm1(o * L) / o if o != 0 else L
            with np.errstate(all="ignore"):
                lead = np.where(L == 0, al / K ** o, al * L / zd)
        return lead * _z_over_x(z, rho) / den * br
    w = f ** o / al
    k = np.log(K / f)
    if model == "expanded":
        A1 = -0.5 * (o - rho * nu * w)
        A2 = (o ** 2 + 3 * (o - rho * nu * w) + (2 - 3 * rho ** 2) * nu ** 2 * w ** 2) / 12
        B = o ** 2 / (24 * w ** 2) + be * rho * nu / (4 * w) + (2 - 3 * rho ** 2) / 24 * nu ** 2
        return (1 + A1 * k + A2 * k ** 2 + B * T) / w
    out = np.empty(T.shape)
    for t in np.unique(T):
        n1, n2, e1, e2 = _term_functions(p, t)
        A1 = (be - 1) / 2 + e1 * w / 2
        A2 = o ** 2 / 12 + (o - e1 * w) / 4 + (4 * n1 + 3 * (e2 - 3 * e1 ** 2)) / 24 * w ** 2
        B = (o ** 2 / 24 + w * be * e1 / 4 + (2 * n2 - 3 * e2) / 24 * w ** 2) / w ** 2
        i = T == t
        out[i] = (1 + A1 * k[i] + A2 * k[i] ** 2 + B * t) / w
    return out


def _black_calls(f, T, K, vol):
    s = vol * np.sqrt(T)
    d = np.log(f / K) / s + 0.5 * s
    cdf = lambda x: 0.5 * np.array([math.erfc(-v / math.sqrt(2.0)) for v in x])
    return f * cdf(d) - K * cdf(d - s)


def _truth(rng, model):
    """Parameters in the ranges of the package's synthetic workloads."""
    u = rng.uniform
    if model in ("hagan", "obloj", "expanded"):
        return [u(0.1, 0.5), u(0.3, 1.0), u(-0.8, 0.2), u(0.2, 1.5)]
    p = [u(0.1, 0.5), u(0.5, 1.0), u(-0.8, 0.0), u(0.2, 1.0), u(0.0, 2.0), u(0.0, 2.0)]
    if model == "dyn2":
        # |rho(t)| <= 0.8 + 0.1 + 0.1 t e^{-at} and nu(t) > 0 hold for a, b >= 0.5
        p[2] = u(-0.7, 0.0)
        p[4], p[5] = u(0.5, 2.0), u(0.5, 2.0)
        p += [u(-0.1, 0.1), u(0.0, 0.2), u(-0.1, 0.1), u(0.0, 0.1)]
    return p


def _maturities(rng, n):
    return np.sort(rng.choice(W.DYN_MATURITIES, n, replace=False))


def _quotes(mats, strikes, lo, hi):
    K = np.linspace(lo, hi, strikes) if strikes > 1 else np.array([1.0])
    return np.repeat(mats, strikes), np.tile(K, len(mats))


def _problem(rng, case, model, prec, T, K, chains):
    """A calibration to the model's own volatilities plus 1e-4 of noise."""
    p = _truth(rng, model)
    vol = _vols(model, p, 1.0, T, K) + rng.normal(0.0, 1e-4, T.size)
    keep = vol > 1e-3  # the expansions can leave the positive range in the far wings
    if not keep.any():
        vol, keep = np.full(T.size, 0.2), np.ones(T.size, dtype=bool)
    lo, hi = BOXES[model]
    return sg.CalibrationProblem(model=MODELS[model], T=T[keep], K=K[keep], market=vol[keep], lo=lo, hi=hi,
                                 prec=PRECS[prec], n_chains=chains, n_levels=case["levels"], chain_len=case["len"],
                                 seed=int(rng.integers(1 << 62)))


def _mc_inputs(case, seed):
    rng = np.random.default_rng(seed)
    T, K = _quotes(W.MC_MATURITIES[: case["mats"]], case["strikes"], 0.6, 1.4)
    p = _truth(rng, case["model"])
    ic = (rng.uniform(size=T.size) < 0.5).astype(np.int8) if case["model"] != "hagan" else np.ones(T.size, np.int8)
    return p, T, K, ic, np.exp(-0.02 * T), int(rng.integers(1 << 62))


CLIQUET = dict(T=1.0, floor_local=-0.02, cap_local=0.02, floor_global=0.0, cap_global=0.2)


def _vol_inputs(case, seed):
    rng = np.random.default_rng(seed)
    T = rng.choice(W.DYN_MATURITIES, case["n"])
    return _truth(rng, case["model"]), T, rng.uniform(0.5, 1.5, case["n"])


def _serving_problems(case, seed):
    rng = np.random.default_rng(seed)
    shape = np.random.default_rng(77)  # the sizes of a case's requests are the case's own
    out = []
    for i in range(case["requests"]):
        mats, strikes = int(shape.integers(1, 13)), int(shape.integers(5, 42))
        if i < case["mc_requests"]:
            T, K = _quotes(W.MC_MATURITIES[: max(1, mats - 4)], strikes, 0.7, 1.3)
            p = _truth(rng, "hagan")
            price = _black_calls(1.0, T, K, np.maximum(_vols("hagan", p, 1.0, T, K), 0.05))
            lo, hi = BOXES["hagan"]
            out.append(sg.CalibrationProblem(model=sg.HAGAN, T=T, K=K, market=np.maximum(price, 1e-6), lo=lo, hi=hi,
                                             cost=sg.COST_MC_PRICE, n_chains=64, n_levels=10, chain_len=10,
                                             mc_paths=case["mc_paths"], mc_steps_per_year=250.0,
                                             mc_seed=int(rng.integers(1 << 62)), seed=int(rng.integers(1 << 62))))
            continue
        model = "hagan" if shape.uniform() < 0.8 else ("dyn1", "dyn2")[int(shape.integers(2))]
        T, K = _quotes(_maturities(shape, mats), strikes, 0.7, 1.3)
        out.append(_problem(rng, case, model, "fp32", T, K, case["chains"]))
    return out


# ---------------------------------------------------------------------------
# What a program has before the call, and the call
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    if kind == "vol":
        p, T, K = _vol_inputs(case, seed)
        return {"kind": kind, "model": MODELS[case["model"]], "p": p, "prec": PRECS[case["prec"]],
                "T": torch.tensor(T, device="cuda"), "K": torch.tensor(K, device="cuda")}
    if kind == "calibrate":
        mats = np.array([1.0]) if case["mats"] == 1 else _maturities(np.random.default_rng(case["mats"]), case["mats"])
        dyn = case["model"].startswith("dyn")
        T, K = _quotes(mats, case["strikes"], 0.5 if dyn else 0.6, 1.5 if dyn else 1.4)
        return {"kind": kind, "problem": _problem(rng, case, case["model"], case["prec"], T, K, case["chains"])}
    if kind == "surface":
        problems = []
        for T1 in W.SURFACE_MATURITIES[: case["smiles"]]:
            T, K = _quotes(np.array([T1]), case["strikes"], 0.5, 1.5)
            problems.append(_problem(rng, case, case["model"], case["prec"], T, K, case["chains"]))
        return {"kind": kind, "plan": sg.Plan(problems)}
    if kind == "mc":
        p, T, K, ic, disc, path_seed = _mc_inputs(case, seed)
        return {"kind": kind, "model": MODELS[case["model"]], "p": p, "T": T, "K": K, "ic": ic, "disc": disc,
                "paths": case["paths"], "spy": float(case["spy"]), "seed": path_seed, "prec": PRECS[case["prec"]],
                "scheme": sg.MC_BESSEL if case["scheme"] == "bessel" else None}
    if kind == "cliquet":
        return {"kind": kind, "model": MODELS[case["model"]], "p": _truth(rng, case["model"]),
                "resets": case["resets"], "paths": case["paths"], "spy": float(case["spy"]),
                "seed": int(rng.integers(1 << 62)), "prec": PRECS[case["prec"]]}
    return {"kind": kind, "problems": _serving_problems(case, seed),
            "server": sg.Server(device_bytes=1 << 28, max_active=64, max_quotes=512)}


def _result(r):
    return {"params": r.params, "misfit": r.misfit, "misfit_fp64": r.misfit_fp64, "restart": r.restart_params,
            "restart_misfit": r.restart_misfit, "counts": np.array([r.n_evals, r.n_accepts, r.status])}


def _results(rs):
    """The results of several calibrations, one array for each field."""
    d = max(len(r.params) for r in rs)
    pad = lambda x: np.pad(np.asarray(x, dtype=np.float64), (0, d - len(x)))
    return {"params": np.stack([pad(r.params) for r in rs]), "restart": np.stack([pad(r.restart_params) for r in rs]),
            "misfit": np.array([r.misfit for r in rs]), "misfit_fp64": np.array([r.misfit_fp64 for r in rs]),
            "restart_misfit": np.array([r.restart_misfit for r in rs]),
            "counts": np.array([[r.n_evals, r.n_accepts, r.status] for r in rs])}


def run(s):
    kind = s["kind"]
    if kind == "vol":
        return sg.implied_vol(s["model"], s["p"], 1.0, s["T"], s["K"], prec=s["prec"])
    if kind == "calibrate":
        return _result(sg.calibrate(s["problem"]))
    if kind == "surface":
        s["plan"].run()
        return _results(s["plan"].results())
    if kind == "mc":
        return sg.mc_price(s["model"], s["p"], 1.0, s["T"], s["K"], is_call=s["ic"], discount=s["disc"],
                           n_paths=s["paths"], steps_per_year=s["spy"], seed=s["seed"], prec=s["prec"],
                           scheme=s["scheme"])
    if kind == "cliquet":
        return sg.mc_cliquet(s["model"], s["p"], 1.0, n_resets=s["resets"], n_paths=s["paths"],
                             steps_per_year=s["spy"], seed=s["seed"], prec=s["prec"], **CLIQUET)
    tickets = [s["server"].submit(p) for p in s["problems"]]
    return _results([s["server"].wait(t, timeout_ms=60000) for t in tickets])


# ---------------------------------------------------------------------------
# What one pass cannot do without
# ---------------------------------------------------------------------------
#: Floating operations of one quote's formula, one maturity's term functions, one path step
_QUOTE = {"hagan": 45, "obloj": 50, "expanded": 7, "dyn1": 7, "dyn2": 7}
_MAT = {"hagan": 0, "obloj": 0, "expanded": 0, "dyn1": 180, "dyn2": 420}
_STEP = {"euler": 30, "bessel": 90}


def _calibration_flops(model, quotes, mats, chains, levels, length):
    return float(chains) * levels * length * (quotes * _QUOTE[model] + mats * _MAT[model] + 40)


def work(case):
    kind = case["kind"]
    if kind == "vol":
        return {"bytes": 24.0 * case["n"], "flops": float(case["n"]) * (_QUOTE[case["model"]] + _MAT[case["model"]] + 20)}
    if kind == "calibrate":
        q = case["mats"] * case["strikes"]
        return {"bytes": 24.0 * q + 200, "flops": _calibration_flops(case["model"], q, case["mats"], case["chains"],
                                                                     case["levels"], case["len"])}
    if kind == "surface":
        return {"bytes": case["smiles"] * (24.0 * case["strikes"] + 200),
                "flops": case["smiles"] * _calibration_flops(case["model"], case["strikes"], 1, case["chains"],
                                                             case["levels"], case["len"])}
    if kind == "mc":
        q = case["mats"] * case["strikes"]
        steps = math.ceil(W.MC_MATURITIES[case["mats"] - 1] * case["spy"])
        return {"bytes": 41.0 * q, "flops": float(case["paths"]) * (steps * _STEP[case["scheme"]] + 5.0 * q)}
    if kind == "cliquet":
        return {"bytes": 200.0, "flops": float(case["paths"]) * math.ceil(case["spy"]) * _STEP["euler"]}
    shape = np.random.default_rng(77)
    b = f = 0.0
    for i in range(case["requests"]):
        mats, strikes = int(shape.integers(1, 13)), int(shape.integers(5, 42))
        if i < case["mc_requests"]:
            mats = max(1, mats - 4)
            f += 64 * 100.0 * case["mc_paths"] * (math.ceil(W.MC_MATURITIES[mats - 1] * 250) * 30 + 5 * mats * strikes)
        else:
            model = "hagan" if shape.uniform() < 0.8 else ("dyn1", "dyn2")[int(shape.integers(2))]
            _maturities(shape, mats)
            f += _calibration_flops(model, mats * strikes, mats, case["chains"], case["levels"], case["len"])
        b += 24.0 * mats * strikes + 200
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# What a call should return, in 64 bits
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c, seed):
    """Philox4x32-10 of Salmon et al. (SC'11) on int64 tensors holding 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    x, y, z, w = c
    for _ in range(10):
        a, b = x * 0xD2511F53, z * 0xCD9E8D57
        x, y, z, w = ((b >> 32) & _M32) ^ y ^ k0, b & _M32, ((a >> 32) & _M32) ^ w ^ k1, a & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return x, y, z, w


def _uniform(w):
    return ((w >> 9).double() + 0.5) * 2.0 ** -23


def _normals(wa, wb):
    r, t = torch.sqrt(-2 * torch.log(_uniform(wa))), 2 * math.pi * _uniform(wb)
    return r * torch.cos(t), r * torch.sin(t)


def _grid(mats, spy):
    """Right end, length and maturity index (or -1) of every step: multiples of 1/spy and the maturities."""
    out, prev, k = [], 0.0, 1
    for m, T in enumerate(mats):
        while k / spy < T - 1e-10:
            out.append((k / spy, k / spy - prev, -1))
            prev = k / spy
            k += 1
        out.append((T, T - prev, m))
        prev = T
        if abs(k / spy - T) <= 1e-10:
            k += 1
    return out


def _nu_rho(p, t):
    p = list(p) + [0.0] * 10
    return (p[3] + p[9] * t) * math.exp(-p[5] * t) + p[7], (p[2] + p[8] * t) * math.exp(-p[4] * t) + p[6]


def _euler_paths(p, mats, spy, n, seed):
    """Forwards at each maturity by the log-Euler scheme of Sec. 4."""
    j = torch.arange(n, device="cuda", dtype=torch.int64)
    zero = torch.zeros_like(j)
    lf = torch.zeros(n, device="cuda", dtype=torch.float64)
    la = torch.full_like(lf, math.log(p[0]))
    dead = torch.zeros(n, device="cuda", dtype=torch.bool)
    for i, (t, h, m) in enumerate(_grid(mats, spy)):
        if i % 2 == 0:
            words = _philox((j, zero + (i >> 1), zero, zero + 0x4D430000), seed)
        z1, z2 = _normals(words[0], words[1]) if i % 2 == 0 else _normals(words[2], words[3])
        nu, rho = _nu_rho(p, t)
        s = torch.exp(la + (p[1] - 1) * lf)
        lf = lf + s * math.sqrt(h) * (rho * z1 + math.sqrt(max(0.0, 1 - rho * rho)) * z2) - 0.5 * h * s * s
        la = la + nu * math.sqrt(h) * z1 - 0.5 * nu * nu * h
        dead = dead | ~(lf >= math.log(1e-12))
        if m >= 0:
            yield torch.where(dead, torch.zeros_like(lf), torch.exp(lf))


def _gamma(a, n, j, i, x, u, ub, seed):
    """Gamma(a) draws by Marsaglia and Tsang's method (ACM TOMS 26(3), 2000), eight trials."""
    ap = a if a >= 1 else a + 1
    d = ap - 1 / 3
    c = 1 / math.sqrt(9 * d)
    g = torch.full((n,), d, device="cuda", dtype=torch.float64)
    todo = torch.arange(n, device="cuda")
    for t in range(8):
        if t:
            zero = torch.zeros_like(todo)
            w = _philox((j[todo], zero + i, zero + (t + 1), zero + 0x4D420000), seed)
            x, u = _normals(w[0], w[1])[0], _uniform(w[2])
        v = (1 + c * x) ** 3
        ok = (v > 0) & ((u < 1 - 0.0331 * x ** 4) | (torch.log(u) < 0.5 * x * x + d * (1 - v + torch.log(v.clamp_min(1e-300)))))
        g[todo[ok]] = d * v[ok]
        todo = todo[~ok]
        if not len(todo):
            break
    return g * ub ** (1 / a) if a < 1 else g


def _bessel_paths(p, mats, spy, n, seed):
    """Forwards at each maturity by the conditional-Bessel step."""
    j = torch.arange(n, device="cuda", dtype=torch.int64)
    zero = torch.zeros_like(j)
    beta = p[1]
    o = 1 - beta
    Y = torch.full((n,), 1 / o, device="cuda", dtype=torch.float64)
    A = torch.full_like(Y, p[0])
    dead = torch.zeros(n, device="cuda", dtype=torch.bool)
    for i, (t, h, m) in enumerate(_grid(mats, spy)):
        w0 = _philox((j, zero + i, zero, zero + 0x4D420000), seed)
        w1 = _philox((j, zero + i, zero + 1, zero + 0x4D420000), seed)
        za, n1 = _normals(w0[0], w0[1])
        n2, x0 = _normals(w0[2], w0[3])
        nu, rho = _nu_rho(p, t)
        kap, q = nu * math.sqrt(h), max(0.0, (1 - rho) * (1 + rho))
        em = torch.expm1(kap * za - 0.5 * kap * kap)
        A1 = A * (1 + em)
        Y0 = Y + A * rho * math.sqrt(h) * (em / kap if kap > 0 else za)
        tau = q * 0.5 * h * (A * A + A1 * A1)
        A = A1
        G = _gamma(0.5 + 0.5 * (beta / o) / q, n, j, i, x0, _uniform(w1[0]), _uniform(w1[1]), seed)
        mm = Y0 * Y0 / (2 * tau)
        dead = dead | ~(Y0 > 0) | ~(G < mm)
        Y = torch.where(dead, torch.ones_like(Y), torch.sqrt(tau * ((n1 + torch.sqrt((2 * (mm - G)).clamp_min(0))) ** 2 + n2 ** 2)))
        if m >= 0:
            yield torch.where(dead, torch.zeros_like(Y), (o * Y) ** (1 / o))


def _mean_and_error(v, disc):
    n = v.numel()
    s, s2 = v.sum(), (v * v).sum()
    mean = s / n
    return disc * mean, disc * torch.sqrt(((s2 - s * mean) / (n - 1)).clamp_min(0) / n)


def exact(case, seed):
    kind = case["kind"]
    if kind == "vol":
        p, T, K = _vol_inputs(case, seed)
        return _vols(case["model"], p, 1.0, T, K)
    if kind == "mc":
        p, T, K, ic, disc, path_seed = _mc_inputs(case, seed)
        mats = np.unique(T)
        paths = _bessel_paths if case["scheme"] == "bessel" else _euler_paths
        price, se = np.empty(T.size), np.empty(T.size)
        for m, F in enumerate(paths(p, mats, float(case["spy"]), case["paths"], path_seed)):
            for q in np.flatnonzero(T == mats[m]):
                x = F - K[q] if ic[q] else K[q] - F
                a, b = _mean_and_error(x.clamp_min(0.0), disc[q])
                price[q], se[q] = float(a), float(b)
        return price, se
    if kind == "cliquet":
        rng = np.random.default_rng(seed)
        p = _truth(rng, case["model"])
        path_seed = int(rng.integers(1 << 62))
        n, prev, total = case["resets"], None, 0.0
        for F in _euler_paths(p, [(i + 1) * CLIQUET["T"] / n for i in range(n)], float(case["spy"]), case["paths"],
                              path_seed):
            if prev is not None:
                R = torch.where(prev > 0, F / torch.where(prev > 0, prev, torch.ones_like(prev)) - 1, torch.zeros_like(F))
                total = total + R.clamp(CLIQUET["floor_local"], CLIQUET["cap_local"])
            prev = F
        a, b = _mean_and_error(total.clamp(CLIQUET["floor_global"], CLIQUET["cap_global"]), 1.0)
        return np.array([float(a)]), np.array([float(b)])
    # a calibration's end point is that of one trajectory of accept / reject
    # decisions in its own precision: there is no 64-bit value to compare with
    return None
