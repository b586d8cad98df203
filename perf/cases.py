"""The work that a user of this package has it do, as cases that can be timed and checked.

A case is one call (or one short run) of a public entry point on seeded inputs:
likelihood batches in both precisions, the allocation-free entry point, mode cross terms,
relative binning, the ensemble sampler, and the flow proposal's evaluation and training.
Sizes are those of the repository's workloads (``workloads.py``, ``bench.py``) and tests.

``exact`` restates the method in plain torch FP64 (waveform, response, not-a-knot splines,
dense sums; relative binning; the flow without its 16-bit operands) and uses nothing of
the package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

DAY_S = 86400.0
YEAR_S = 3.15576e7
TWO_PI = 2.0 * math.pi
MSUN_S = 4.925490947641267e-06
CLIGHT = 299792458.0
GPC_S = 3.0856775814913673e25 / CLIGHT
AU_S = 1.495978707e11 / CLIGHT
ARM_S = 2.5e9 / CLIGHT
X_JOIN, X_CUT = 0.018, 0.2
MODES = ((2, 2), (3, 3), (4, 4), (2, 1), (3, 2), (4, 3))

# frequency grids by name: f_min, f_max, observation time, t_coal - t_ref
GRIDS = {
    "month": (1e-4, 1e-2, 30.0 * DAY_S, 30.0 * DAY_S),    # the one-walker workload
    "month_wide": (1e-4, 2e-2, 30.0 * DAY_S, 30.0 * DAY_S),
    "quarter": (3e-5, 4.1e-2, 91.3 * DAY_S, 91.3 * DAY_S),
    "year": (1e-5, 1e-1, YEAR_S, YEAR_S),                 # the benchmark's grid
}
# injections: M_T, q, a1, a2, z or D_L, phi_ref, iota, lambda, beta, psi, t_ref
MONTH_INJECTION = (1e6, 0.2, 0.0, 0.0, 6.79, 1.0, math.pi / 3, 1.0, 0.3, 0.5, 1000.0)
YEAR_INJECTION = (2e6, 1 / 3, 0.0, 0.0, 36.59, 2.14, 1.05, -0.024, 0.62, 2.03, 50.25)
SAMPLER_INJECTION = (2e6, 0.5, 0.0, 0.0, 26.0, 2.14, 1.05, -0.024 % TWO_PI, 0.62, 2.03, 3600.0)
# the Table II binaries whose mode content the paper breaks down
TABLE2 = (
    (2e6, 1 / 3, 0.0, 0.0, 36.59, 2.14, 1.05, -0.024, 0.62, 2.03, 50.25),
    (2e6, 1 / 3, 0.85, 0.88, 36.59, 2.14, 1.05, -0.024, 0.62, 2.03, 50.25),
    (2e6, 1 / 3, -0.83, -0.89, 36.59, 2.14, 1.05, -0.024, 0.62, 2.03, 50.25),
    (4e7, 1 / 5, 0.0, 0.0, 15.93, 3.10, 1.34, 4.21, -0.73, 0.14, 23.93),
    (3e5, 7 / 10, 0.0, 0.0, 70.58, 1.22, 1.32, 2.24, -0.22, 2.73, 94.33),
)
# prior box of the sampling coordinates (Table I)
LOWER = np.array([math.log(1e3), 0.05, -0.99, -0.99, math.log(0.044), 0.0, -1.0, 0.0, -1.0, 0.0, 0.0])
UPPER = np.array([math.log(1e9), 1.0, 0.99, 0.99, math.log(1298.0), TWO_PI, 1.0, TWO_PI, 1.0,
                  math.pi, math.log(3.15576e8)])
FLOW_C, FLOW_H, FLOW_D = 8, 128, 11


def listed():
    like = {"kind": "loglike", "api": "device", "bad": 0.0, "graph": False, "near": False}
    return [
        # the smallest call there is: one walker, one mode, host buffers in and out
        dict(like, name="one_22_month", api="host", precision="fp64", walkers=1, modes=1, knots=256,
             grid="month", logm_lo=6.0, logm_hi=6.0),
        # one walker on the full grid from code that may not allocate
        dict(like, name="one_noalloc_year", api="noalloc", precision="fp64", walkers=1, modes=6,
             knots=1024, grid="year", logm_lo=5.9, logm_hi=6.6),
        # an uneven batch: odd counts, masses over six decades, some walkers outside the
        # physical range, bands of very different lengths
        dict(like, name="ragged_37_quarter", precision="fp64", walkers=37, modes=4, knots=509,
             grid="quarter", logm_lo=3.0, logm_hi=9.0, bad=0.1),
        # the benchmark: 1024 prior draws on the 1-yr grid, in both precisions (split
        # precision is what samplers run on: as they do, its cases ask for ln L alone)
        dict(like, name="prior_1024_fp64", precision="fp64", walkers=1024, modes=6, knots=1024,
             grid="year", logm_lo=5.0, logm_hi=7.0),
        dict(like, name="prior_1024_split", precision="split", walkers=1024, modes=6, knots=1024,
             grid="year", logm_lo=5.0, logm_hi=7.0),
        # half a step of the 8 x 256 sampler: 1024 proposals near the posterior, those that
        # left the prior box marked invalid, replayed as a graph
        dict(like, name="posterior_1024_split", precision="split", walkers=1024, modes=6, knots=1024,
             grid="year", logm_lo=6.3, logm_hi=6.3, bad=0.15, graph=True, near=True),
        # the largest batch: 8192 walkers over the whole mass range
        dict(like, name="wide_8192_split", precision="split", walkers=8192, modes=6, knots=1024,
             grid="year", logm_lo=3.0, logm_hi=9.0),
        # relative binning of 1024 walkers about a fiducial
        {"kind": "rb", "name": "rb_1024_year", "walkers": 1024, "modes": 6, "bins": 256, "grid": "year"},
        # mode-by-mode breakdown with cross terms of five injections (21 passes)
        {"kind": "cross", "name": "cross_5_year", "precision": "fp64", "walkers": 5, "modes": 6,
         "knots": 1024, "grid": "year"},
        # the parallel-tempered sampler on a month of data
        {"kind": "sampler", "name": "sampler_4x64_month", "temps": 4, "walkers": 64, "modes": 2,
         "knots": 256, "grid": "month", "steps": 20},
        # the flow's part of a sampler step: 256 proposals and the density of 256 walkers
        {"kind": "flow", "name": "flow_256", "rows": 256},
        # training on the coldest chain: 1024-row minibatches
        {"kind": "train", "name": "train_1024", "rows": 12800, "batch": 1024, "iters": 40},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loglike"] * 5 + ["rb", "cross", "sampler", "flow", "train"])
    if kind == "loglike":
        case = {"kind": kind, "modes": rng.randint(1, 6), "knots": rng.choice([256, 333, 509, 777, 1024]),
                "bad": rng.choice([0.0, 0.0, 0.1]), "graph": rng.random() < 0.3, "near": rng.random() < 0.3}
        if rng.random() < 0.4:  # split precision: large batches on the full grid
            center, half = rng.uniform(5.3, 6.7), rng.uniform(0.0, 0.8)
            case.update(precision="split", api="device", grid="year", walkers=_log_int(rng, 64, 2000))
        else:
            center, half = rng.uniform(5.0, 7.5), rng.uniform(0.0, 1.5)
            case.update(precision="fp64", api=rng.choice(["device", "device", "host", "noalloc"]),
                        grid=rng.choice(["month", "month_wide", "quarter", "year"]),
                        walkers=_log_int(rng, 1, 400))
        case.update(logm_lo=round(center - half, 2), logm_hi=round(center + half, 2))
        if case["api"] == "noalloc":  # the entry point's own limits
            case["graph"] = False
            case["walkers"] = max(1, min(4 if case["grid"] == "year" else 9, case["walkers"],
                                         8192 // (case["modes"] * case["knots"])))
        return case
    if kind == "rb":
        return {"kind": kind, "walkers": _log_int(rng, 1, 1500), "modes": rng.randint(1, 6),
                "bins": rng.choice([64, 100, 128, 200, 256]), "grid": rng.choice(["month", "year"])}
    if kind == "cross":
        return {"kind": kind, "precision": "fp64", "walkers": rng.randint(1, 5),
                "modes": rng.randint(2, 6), "knots": rng.choice([256, 511, 1024]),
                "grid": rng.choice(["month", "quarter", "year"])}
    if kind == "sampler":
        return {"kind": kind, "temps": rng.randint(1, 8), "walkers": 8 * rng.randint(1, 16),
                "modes": rng.randint(1, 3), "knots": rng.choice([128, 256]), "grid": "month",
                "steps": rng.randint(5, 25)}
    if kind == "flow":
        return {"kind": kind, "rows": _log_int(rng, 1, 20000)}
    return {"kind": kind, "rows": _log_int(rng, 500, 60000), "batch": 64 * _log_int(rng, 1, 32),
            "iters": rng.randint(5, 50)}


# ------------------------------------------------------------------------------ inputs

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=_dev())


def _grid(case):
    lo, hi, T, t0 = GRIDS[case["grid"]]
    df = 1.0 / T
    return lo, df, int(math.floor((hi - lo) / df)) + 1, t0


def _distance(z):
    """D_L [Gpc] of a flat universe, H0 = 67.7, Om = 0.31 (only to draw sensible loudness)."""
    zz = np.linspace(0.0, 10.0, 20001)
    e = 1.0 / np.sqrt(0.31 * (1.0 + zz) ** 3 + 0.69)
    c = np.concatenate([[0.0], np.cumsum(0.5 * (e[1:] + e[:-1]) * np.diff(zz))])
    return (1.0 + z) * 299792.458 / 67.7 / 1000.0 * np.interp(z, zz, c)


def _near(theta, B, rng, scale):
    th = np.asarray(theta)[None, :] * (1.0 + scale * rng.standard_normal((B, 11)))
    th[:, 1] = np.minimum(th[:, 1], 1.0)
    th[:, 2:4] = np.clip(scale * 10.0 * rng.standard_normal((B, 2)) + np.asarray(theta)[2:4], -0.99, 0.99)
    return th


def _walkers(case, seed):
    rng = np.random.default_rng([seed, 17])
    B = case["walkers"]
    if case["kind"] == "cross":
        return np.array(TABLE2[:B]) * (1.0 + 1e-3 * rng.standard_normal((B, 11)))
    if case["kind"] == "rb":
        return _near(_injection(case), B, rng, 2e-4)
    if case["near"]:  # around the injection
        th = _near(_injection(case), B, rng, 1e-3)
    else:
        th = np.empty((B, 11))
        th[:, 0] = 10.0 ** rng.uniform(case["logm_lo"], case["logm_hi"], B)
        th[:, 1] = rng.uniform(0.05, 1.0, B)
        th[:, 2:4] = rng.uniform(-0.99, 0.99, (B, 2))
        th[:, 4] = _distance(rng.uniform(1.0, 8.0, B))
        th[:, 5] = rng.uniform(0.0, TWO_PI, B)
        th[:, 6] = np.arccos(rng.uniform(-1.0, 1.0, B))
        th[:, 7] = rng.uniform(0.0, TWO_PI, B)
        th[:, 8] = np.arcsin(rng.uniform(-1.0, 1.0, B))
        th[:, 9] = rng.uniform(0.0, math.pi, B)
        th[:, 10] = rng.uniform(0.0, 3600.0, B)
    bad = rng.random(B) < case["bad"]  # as the sampler marks proposals outside the prior
    th[bad, 0] = np.nan
    return th


def _injection(case):
    if case["grid"] != "year":
        return np.array(MONTH_INJECTION)
    return np.array(SAMPLER_INJECTION if case["kind"] == "rb" or case.get("near") else YEAR_INJECTION)


def _freqs(f0, df, n):
    return f0 + torch.arange(n, dtype=torch.float64, device=_dev()) * df


def _psd(f):
    """One-sided A, E, T noise of first-generation channels with equal arms, [3, n]."""
    om = TWO_PI * f
    conv = (om / CLIGHT) ** 2
    oms = 2.25e-22 * (1.0 + (2e-3 / f) ** 4) * conv
    acc = 9e-30 * (1.0 + (0.4e-3 / f) ** 2) * (1.0 + (f / 8e-3) ** 4) / om ** 4 * conv
    x = om * ARM_S
    s2, c = torch.sin(x) ** 2, torch.cos(x)
    ae = 8.0 * s2 * ((2.0 + c) * oms + 2.0 * (3.0 + 2.0 * c + torch.cos(2.0 * x)) * acc)
    t = 16.0 * s2 * (1.0 - c) * (oms + 2.0 * (1.0 - c) * acc)
    return torch.stack([ae, ae, t])


def _data(case, seed):
    """f0, df, n, t0, the data [3, n, 2] (injection plus coloured noise) and the PSD [3, n]."""
    f0, df, n, t0 = _grid(case)
    psd = _psd(_freqs(f0, df, n))
    gen = torch.Generator(device=_dev()).manual_seed(1000003 * seed + 7)
    d = torch.randn((3, n, 2), generator=gen, dtype=torch.float64, device=_dev())
    d *= (0.5 * torch.sqrt(psd / df))[:, :, None]
    inj = np.array(_injection(case))
    inj[4] *= 1.0 + 0.2 * np.random.default_rng([seed, 3]).random()
    # amplitudes and phases of the injected signal from its own splines
    tm = _Template(inj[None, :], MODES, 1024, f0, df, n, t0)
    for jl, h in tm.modes_of(0):
        if h is not None:
            d[:, jl:jl + h.shape[1]] += h
    return f0, df, n, t0, d, psd


def _config(case):
    from paper_2005_01827_gb300 import lisalike as LL

    cfg = LL.lisa_like_default_config()
    cfg.n_modes, cfg.n_knots, cfg.t0_s = case["modes"], case["knots"], GRIDS[case["grid"]][3]
    for k, (l, m) in enumerate(MODES[:case["modes"]]):
        cfg.modes[k][0], cfg.modes[k][1] = l, m
    return cfg


def _handle(case, seed, B):
    import paper_2005_01827_gb300 as pkg

    f0, df, n, t0, d, psd = _data(case, seed)
    prec = pkg.LISA_PREC_SPLIT if case.get("precision") == "split" else pkg.LISA_PREC_FP64
    like = pkg.LisaLike(modes=MODES[:case["modes"]], n_knots=case.get("knots", 128), precision=prec,
                        t0=t0, max_batch=B)
    like.set_data(f0, df, n, d.cpu().numpy(), psd.cpu().numpy())
    return like


def _flow_weights(seed, scale=0.05):
    """A flow that does something: random hidden layers, a small output layer."""
    rng = np.random.default_rng([seed, 5])
    C, H, D = FLOW_C, FLOW_H, FLOW_D

    def u(lim, *shape):
        return rng.uniform(-lim, lim, shape).astype(np.float32)

    l1, l2 = math.sqrt(6.0 / D), math.sqrt(6.0 / H)
    return {"W1": u(l1, C, H, D), "b1": u(0.1, C, H), "W2": u(l2, C, H, H), "b2": u(0.1, C, H),
            "W3": u(scale * l2, C, 2 * D, H), "b3": u(0.05, C, 2 * D)}


def _chain(seed, n):
    """Sampling coordinates of a posterior: correlated, of very different widths, one bent."""
    rng = np.random.default_rng([seed, 9])
    sig = np.array([1e-3, 2e-3, 1e-2, 2e-2, 5e-2, 0.3, 4e-2, 1e-2, 1e-2, 0.2, 1e-4])
    A = np.eye(11) + 0.4 * rng.standard_normal((11, 11))
    g = rng.standard_normal((n, 11)) @ A.T
    g[:, 5] += 0.3 * (g[:, 4] ** 2 - 1.0)
    mu = np.array([14.5, 0.5, 0.1, -0.1, 3.3, 2.1, 0.5, 3.0, 0.5, 1.5, 8.2])
    return mu + sig * g


def _whitening(x):
    mu = x.mean(axis=0)
    c = (x - mu).T @ (x - mu) / x.shape[0]
    return mu, np.linalg.cholesky(c)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "loglike":
        th = _walkers(case, seed)
        B = th.shape[0]
        if case["api"] == "noalloc":
            f0, df, n, t0, d, psd = _data(case, seed)
            w = 4.0 * df / psd
            cols = [w[0], w[1], w[2]]
            for c in range(3):
                cols += [w[c] * d[c, :, 0], w[c] * d[c, :, 1]]
            dd = float((w[:, :, None] * d * d).sum())
            return {"case": case, "cfg": _config(case), "f0": f0, "df": df, "n": n, "dd": dd,
                    "bins": torch.stack(cols, dim=1).contiguous(), "P": _t(th), "B": B,
                    "out": torch.empty((3, B), dtype=torch.float64, device=_dev())}
        like = _handle(case, seed, B)
        if case["graph"]:
            from paper_2005_01827_gb300 import lisalike as LL

            LL.lisa_like_set_graphs(like.h, True)
        return {"case": case, "like": like, "th": th, "P": _t(th), "B": B,
                "out": torch.empty((3, B), dtype=torch.float64, device=_dev())}
    if kind == "rb":
        th = _walkers(case, seed)
        like = _handle(case, seed, th.shape[0])
        like.set_fiducial(_injection(case), case["bins"])
        return {"case": case, "like": like, "P": _t(th), "B": th.shape[0],
                "out": torch.empty((3, th.shape[0]), dtype=torch.float64, device=_dev())}
    if kind == "cross":
        return {"case": case, "like": _handle(case, seed, case["walkers"]), "th": _walkers(case, seed)}
    if kind == "sampler":
        from paper_2005_01827_gb300 import lisalike as LL

        T, W, t0 = case["temps"], case["walkers"], GRIDS[case["grid"]][3]
        like = _handle(case, seed, T * W // 2)
        s = LL.LisaSampler(like, n_temps=T, n_walkers=W, seed=seed + 1, lower=LOWER, upper=UPPER)
        xc = LL.from_physical(np.array(MONTH_INJECTION), True, t0)
        scale = np.array([1e-3, 1e-2, 1e-2, 1e-2, 1e-2, 1e-1, 1e-2, 1e-3, 1e-3, 1e-2, 1e-4])
        s.set_state(LL.sky_mode_init(xc, scale, LOWER, UPPER, T, W, seed + 11))
        return {"case": case, "like": like, "sampler": s}
    from paper_2005_01827_gb300 import lisalike as LL

    flow = LL.Flow(seed=1)
    w = _flow_weights(seed)
    flow.set_weights(w)
    x = _chain(seed, case["rows"] + 64)
    if kind == "flow":
        mu, L = _whitening(_chain(seed + 1, 4000))
        flow.set_whitening(mu, L)
        n = case["rows"]
        z = np.random.default_rng([seed, 21]).standard_normal((n, 11))
        e = lambda *s: torch.empty(s, dtype=torch.float64, device=_dev())  # noqa: E731
        return {"case": case, "flow": flow, "z": _t(z), "x": _t(x[:n]), "n": n,
                "y": e(n, 11), "qy": e(n), "u": e(n, 11), "qx": e(n)}
    return {"case": case, "flow": flow, "w": LL.pack_flow_weights(w), "data": _t(x[:case["rows"]])}


# ------------------------------------------------------------------------------ one pass

def _stream():
    return torch.cuda.current_stream().cuda_stream


def run(state):
    from paper_2005_01827_gb300 import lisalike as LL

    case = state["case"]
    kind = case["kind"]
    if kind == "loglike":
        if case["api"] == "host":
            return state["like"].loglike(state["th"])
        o = state["out"]
        if case["api"] == "noalloc":
            LL.lisa_like_loglike_noalloc(state["cfg"], state["f0"], state["df"], state["n"],
                                         state["bins"], state["dd"], state["P"], state["B"], o[0],
                                         o[1], o[2], _stream())
        elif case["precision"] == "split":
            LL.lisa_like_loglike_device(state["like"].h, state["P"], state["B"], o[0], stream=_stream())
            return o[0]
        else:
            LL.lisa_like_loglike_device(state["like"].h, state["P"], state["B"], o[0], o[1], o[2],
                                        _stream())
        return o[0], o[1], o[2]
    if kind == "rb":
        o = state["out"]
        LL.lisa_like_loglike_rb_device(state["like"].h, state["P"], state["B"], o[0], o[1], o[2],
                                       _stream())
        return o[0], o[1], o[2]
    if kind == "cross":
        return state["like"].mode_cross(state["th"])
    if kind == "sampler":
        chain, lnl = state["sampler"].run(case["steps"])
        x, l, betas, _ = state["sampler"].state()
        acc, swaps = state["sampler"].counts()
        return {"chain": chain, "chain_lnl": lnl, "x": x, "lnl": l, "betas": betas, "acc": acc,
                "swaps": swaps}
    if kind == "flow":
        lib, f, n, s = LL.load(), state["flow"], state["n"], _stream()
        p = LL._ptr
        LL._fcheck(lib.lisa_flow_generate(f.h, p(state["z"]), n, p(state["y"]), p(state["qy"]), s), f.h)
        LL._fcheck(lib.lisa_flow_normalize(f.h, p(state["x"]), n, p(state["u"]), p(state["qx"]), s), f.h)
        return {k: state[k] for k in ("y", "qy", "u", "qx")}
    f = state["flow"]
    f.set_weights(state["w"])
    loss = f.train(state["data"], case["iters"], batch=case["batch"])
    return {"loss": loss, "weights": f.weights()}


def _active_bins(case, seed=0):
    """(walker, mode, bin) and (walker, bin) counts from the ringdown cut and the start of
    the band at leading order: what the sums of one pass run over."""
    f0, df, n, t0 = _grid(case)
    th = _walkers(case, seed)
    ok = np.isfinite(th[:, 0])
    M = np.where(ok, th[:, 0], 1.0) * MSUN_S
    eta = th[:, 1] / (1.0 + th[:, 1]) ** 2
    flow22 = (t0 / (5.0 / 256.0 * M / eta * (math.pi * M) ** (-8.0 / 3.0))) ** (-3.0 / 8.0)
    tot, union = 0.0, 0.0
    lo_u, hi_u = np.full(M.shape, np.inf), np.zeros(M.shape)
    for (_, m) in MODES[:case["modes"]]:
        lo = np.maximum(f0, 0.5 * m * flow22)
        hi = np.minimum(f0 + (n - 1) * df, 0.5 * m * X_CUT / M)
        c = np.where(ok, np.maximum(0.0, (hi - lo) / df), 0.0)
        tot += c.sum()
        lo_u, hi_u = np.where(c > 0, np.minimum(lo, lo_u), lo_u), np.where(c > 0, np.maximum(hi, hi_u), hi_u)
    union = np.where(ok & (hi_u > lo_u), (hi_u - lo_u) / df, 0.0).sum()
    return float(tot), float(union), n


def work(case):
    """Bytes: parameters, data and results once.  Operations: per (walker, mode, bin) the
    eight cubics, e^{i phi}'s rotation, the three complex products (75), per (walker, bin)
    the integrand (25); per knot or edge the waveform and response (700)."""
    kind = case["kind"]
    if kind in ("loglike", "cross"):
        mb, wb, n = _active_bins(case)
        B, L, K = case["walkers"], case["modes"], case["knots"]
        passes = 1.0
        if kind == "cross":  # every pair of modes needs its products once
            passes = 1.0
            mb, wb = mb, wb * L * (L + 1) / 2
        bin_bytes = 36.0 if case.get("precision") == "split" else 72.0
        used = min(float(n), wb) if wb else 1.0
        return {"bytes": bin_bytes * used + 8.0 * B * 14,
                "flops": passes * (75.0 * mb + 25.0 * wb) + 700.0 * B * L * K}
    if kind == "rb":
        B, L, E = case["walkers"], case["modes"], case["bins"] + 7
        P = L * (L + 1) // 2
        return {"bytes": 8.0 * E * 6 * (L + 2 * L + 2 * P) + 8.0 * B * 14,
                "flops": B * E * (780.0 * L + 3 * (12.0 * L + 30.0 * P))}
    if kind == "sampler":
        T, W, S = case["temps"], case["walkers"], case["steps"]
        mb, wb, n = _active_bins(dict(case, kind="loglike", walkers=T * W, near=True, bad=0.0))
        return {"bytes": 72.0 * n + 8.0 * T * W * 14 * S,
                "flops": S * (75.0 * mb + 25.0 * wb + 700.0 * T * W * case["modes"] * case["knots"])}
    net = 2.0 * FLOW_H * (FLOW_D + FLOW_H + 2 * FLOW_D)  # one coupling of one row
    wbytes = 2.0 * FLOW_C * FLOW_H * (FLOW_D + FLOW_H + 2 * FLOW_D)
    if kind == "flow":
        return {"bytes": wbytes + 2 * case["rows"] * 8.0 * 23, "flops": 2 * case["rows"] * FLOW_C * net}
    rows = case["iters"] * case["batch"]
    return {"bytes": case["iters"] * 10.0 * wbytes + rows * 88.0 + case["rows"] * 88.0,
            "flops": 3.0 * rows * FLOW_C * net}


# ------------------------------------------------------------------------------ exact values

def _source(th, t0):
    """Constants of the stand-in waveform for parameter rows th [B, 11] (numpy), tensors [B]."""
    ok = np.isfinite(th).all(axis=1)
    p = np.where(ok[:, None], th, np.array(MONTH_INJECTION))
    ok &= (p[:, 0] > 0) & (p[:, 1] > 0) & (p[:, 1] <= 1) & (np.abs(p[:, 2]) <= 0.99) & \
        (np.abs(p[:, 3]) <= 0.99) & (p[:, 4] > 0)
    p = _t(np.where(ok[:, None], p, np.array(MONTH_INJECTION)))
    mt, q, a1, a2, dl = (p[:, i] for i in range(5))
    s = {"ok": ok, "M": mt * MSUN_S, "eta": q / (1 + q) ** 2, "dlt": (1 - q) / (1 + q)}
    eta = s["eta"]
    chis, chia, chieff = 0.5 * (a1 + a2), 0.5 * (a1 - a2), (a1 + q * a2) / (1 + q)
    s.update(phiref=p[:, 5], iota=p[:, 6], lam=p[:, 7], beta=p[:, 8], psi=p[:, 9], tc=p[:, 10] + t0)
    s["amp0"] = torch.sqrt(2 * eta / 3) * math.pi ** (-1 / 6) * s["M"] ** 2 / (dl * GPC_S)
    s["al2"] = -323 / 224 + 451 / 168 * eta
    s["al3"] = (27 / 8 - 11 / 6 * eta) * chis + 27 / 8 * s["dlt"] * chia
    s["ps2"] = 3715 / 756 + 55 / 9 * eta
    s["ps3"] = (113 / 3 - 76 / 3 * eta) * chis + 113 / 3 * s["dlt"] * chia
    af = (2 * math.sqrt(3) * eta - 3.871 * eta ** 2 + 4.028 * eta ** 3 + 0.3 * chieff).clamp(-0.99, 0.99)
    s["xrd"] = (1 - 0.63 * (1 - af) ** 0.3) / (TWO_PI * (1 - 0.0572 * eta - 0.498 * eta ** 2))
    xj = torch.full_like(eta, X_JOIN)
    pj, dj, d2j = _inspiral(s, xj)
    s["phj"], s["c2"] = pj, -0.5 * X_JOIN ** 3 * d2j
    s["c1"] = dj - s["c2"] / X_JOIN ** 2
    lo, hi = 0.25 * s["xrd"], 2.0 * s["xrd"]

    def peak(x):
        v = (math.pi * x) ** (1 / 3)
        r6 = (x / s["xrd"]) ** 6
        return 5 / 6 + 2 / 3 * s["al2"] * v ** 2 + s["al3"] * v ** 3 - 6 * r6 / (1 + r6)

    at_lo, at_hi = peak(lo) <= 0, peak(hi) >= 0
    xl, xh = lo.clone(), hi.clone()
    for _ in range(60):
        mid = 0.5 * (xl + xh)
        up = peak(mid) > 0
        xl, xh = torch.where(up, mid, xl), torch.where(up, xh, mid)
    s["xpk"] = torch.where(at_lo, lo, torch.where(at_hi, hi, 0.5 * (xl + xh)))
    s["phpk"], s["dphpk"] = _phase_slope(s, s["xpk"])
    return s


def _inspiral(s, x):
    v = (math.pi * x) ** (1 / 3)
    k = 1 / (128 * s["eta"])
    a, b, c = v ** -5, s["ps2"] * v ** -3, s["ps3"] * v ** -2
    return (-3 * k * (a + b + c), k / x * (5 * a + 3 * b + 2 * c),
            -k / x ** 2 * (40 / 3 * a + 6 * b + 10 / 3 * c))


def _phase_slope(s, x):
    p, d, _ = _inspiral(s, x)
    late = x > X_JOIN
    return (torch.where(late, s["phj"] + s["c1"] * (x - X_JOIN) - s["c2"] * (1 / x - 1 / X_JOIN), p),
            torch.where(late, s["c1"] + s["c2"] / x ** 2, d))


def _time(s, m, f):
    _, d = _phase_slope(s, 2 * s["M"] * f / m)
    return s["tc"] - s["M"] / TWO_PI * (d - s["dphpk"])


def _col(s):
    """The source constants as columns, to be used against rows of frequencies."""
    return {k: (v[:, None] if isinstance(v, torch.Tensor) else v) for k, v in s.items()}


def _amp_phase(s, l, m, f):
    x = 2 * s["M"] * f / m
    v = (math.pi * x) ** (1 / 3)
    d, e = s["dlt"], s["eta"]
    r = {(2, 2): 1.0, (3, 3): 0.75 * math.sqrt(15 / 14) * d * v,
         (4, 4): 8 / 9 * math.sqrt(5 / 7) * (1 - 3 * e) * v ** 2, (2, 1): math.sqrt(2) / 3 * d * v,
         (3, 2): 1 / 3 * math.sqrt(5 / 7) * (1 - 3 * e) * v ** 2,
         (4, 3): 9 / (4 * math.sqrt(70)) * d * (1 - 2 * e) * v ** 3}[(l, m)]
    off = {(3, 3): -0.5, (4, 4): 1.0, (2, 1): 0.5, (4, 3): -0.5}.get((l, m), 0.0) * math.pi
    p, _ = _phase_slope(s, x)
    a = r * math.sqrt(2 / m) * s["amp0"] * x ** (-7 / 6) * torch.exp(s["al2"] * v ** 2 + s["al3"] * v ** 3)
    return a / (1 + (x / s["xrd"]) ** 6), 0.5 * m * (p - s["phpk"] - s["dphpk"] * (x - s["xpk"])) + off


def _ylm(l, m, th, ph):
    c, s, ct = torch.cos(th / 2), torch.sin(th / 2), torch.cos(th)
    v = {(2, 2): math.sqrt(5 / (4 * math.pi)) * c ** 4, (2, -2): math.sqrt(5 / (4 * math.pi)) * s ** 4,
         (2, 1): math.sqrt(5 / math.pi) * c ** 3 * s, (2, -1): math.sqrt(5 / math.pi) * s ** 3 * c,
         (3, 3): -math.sqrt(21 / (2 * math.pi)) * c ** 5 * s,
         (3, -3): math.sqrt(21 / (2 * math.pi)) * s ** 5 * c,
         (3, 2): 0.5 * math.sqrt(7 / math.pi) * c ** 4 * (3 * ct - 2),
         (3, -2): 0.5 * math.sqrt(7 / math.pi) * s ** 4 * (3 * ct + 2),
         (4, 4): 3 * math.sqrt(7 / math.pi) * c ** 6 * s ** 2,
         (4, -4): 3 * math.sqrt(7 / math.pi) * s ** 6 * c ** 2,
         (4, 3): -3 * math.sqrt(7 / (2 * math.pi)) * c ** 5 * s * (2 * ct - 1),
         (4, -3): 3 * math.sqrt(7 / (2 * math.pi)) * s ** 5 * c * (2 * ct + 1)}[(l, m)]
    return torch.polar(torch.ones_like(v), m * ph) * v


def _response(s, l, m, f):
    """t-dependent A, E, T transfer [3, ...] (complex) and the delay phase of mode (l, m)."""
    t = _time(s, m, f)
    yp, ym = _ylm(l, m, s["iota"], s["phiref"]), _ylm(l, -m, s["iota"], s["phiref"])
    ypc = (-1.0) ** l * yp.conj()
    kp, kc = 0.5 * (ym + ypc), 0.5j * (ym - ypc)
    sl, cl, sb, cb = (g(s[k]) for k in ("lam", "beta") for g in (torch.sin, torch.cos))
    s2, c2 = torch.sin(2 * s["psi"]), torch.cos(2 * s["psi"])
    u, w = (sl, -cl, torch.zeros_like(sl)), (-sb * cl, -sb * sl, cb)
    k = (-cb * cl, -cb * sl, -sb)
    al = TWO_PI * t / YEAR_S
    pre = ARM_S / (4 * math.sqrt(3))
    q = []
    for i in range(3):
        b = TWO_PI * i / 3
        q.append((pre * (torch.cos(2 * al - b) - 3 * math.cos(b)),
                  pre * (torch.sin(2 * al - b) - 3 * math.sin(b)),
                  -2 * math.sqrt(3) * pre * torch.cos(al - b)))
    delay = -TWO_PI * f * AU_S * (k[0] * torch.cos(al) + k[1] * torch.sin(al))
    pfl = math.pi * f * ARM_S
    y = {}
    for a, c in ((0, 1), (0, 2), (1, 2)):
        n = [(q[c][i] - q[a][i]) / ARM_S for i in range(3)]
        un, wn = sum(u[i] * n[i] for i in range(3)), sum(w[i] * n[i] for i in range(3))
        ep, ec = un * un - wn * wn, 2 * un * wn
        F = kp * (c2 * ep + s2 * ec) + kc * (c2 * ec - s2 * ep)
        kn = sum(k[i] * n[i] for i in range(3))
        kq = sum(k[i] * (q[a][i] + q[c][i]) for i in range(3))
        e = -1j * pfl * F * torch.exp(-1j * math.pi * f * (ARM_S + kq))
        y[a, c] = torch.sinc(f * ARM_S * (1 - kn)) * e
        y[c, a] = torch.sinc(f * ARM_S * (1 + kn)) * e
    D = torch.exp(-2j * pfl)
    X, Y, Z = ((1 - D * D) * (y[i2, i0] + D * y[i0, i2] - y[i1, i0] - D * y[i0, i1])
               for i0, i1, i2 in ((0, 1, 2), (1, 2, 0), (2, 0, 1)))
    return torch.stack([(Z - X) / math.sqrt(2), (X - 2 * Y + Z) / math.sqrt(6),
                        (X + Y + Z) / math.sqrt(3)]), delay


def _bands(s, m, f0, df, n):
    """active, f_lo, f_hi, j_lo, j_hi of a mode for every walker (numpy)."""
    M = s["M"]
    fmx = f0 + (n - 1) * df
    hi = torch.clamp(0.5 * m * X_CUT / M, max=fmx)
    fmn = torch.full_like(M, f0)
    act = hi > f0 * (1 + 1e-12)
    from_start = _time(s, m, fmn) >= 0
    act &= from_start | (_time(s, m, hi) >= 0)
    a, c = fmn.clone(), hi.clone()
    for _ in range(60):
        mid = 0.5 * (a + c)
        neg = _time(s, m, mid) < 0
        a, c = torch.where(neg, mid, a), torch.where(neg, c, mid)
    lo = torch.where(from_start, fmn, c)
    act &= hi > lo * (1 + 1e-12)
    jl = torch.clamp(torch.ceil((lo - f0) / df - 1e-9), min=0)
    jh = torch.clamp(torch.floor((hi - f0) / df + 1e-9), max=n - 1)
    act &= jl <= jh
    act = act.cpu().numpy() & s["ok"]
    return act, lo, hi, jl.cpu().numpy(), jh.cpu().numpy()


def _spline(x, y):
    """Not-a-knot cubic coefficients [4, S, Q, K - 1] of y [S, Q, K] on knots x [S, K]."""
    K = x.shape[1]
    h = x[:, 1:] - x[:, :-1]
    sl = (y[:, :, 1:] - y[:, :, :-1]) / h[:, None]
    rhs = 6 * (sl[:, :, 1:] - sl[:, :, :-1])
    dia, sup, sub = 2 * (h[:, :-1] + h[:, 1:]), h[:, 1:].clone(), h[:, :-1].clone()
    dia[:, 0] += h[:, 0] * (h[:, 0] + h[:, 1]) / h[:, 1]
    sup[:, 0] -= h[:, 0] ** 2 / h[:, 1]
    dia[:, -1] += h[:, -1] * (h[:, -2] + h[:, -1]) / h[:, -2]
    sub[:, -1] -= h[:, -1] ** 2 / h[:, -2]
    n = K - 2
    cp = [sup[:, 0] / dia[:, 0]]
    rp = [rhs[:, :, 0] / dia[:, 0, None]]
    for i in range(1, n):
        den = dia[:, i] - sub[:, i] * cp[-1]
        cp.append(sup[:, i] / den)
        rp.append((rhs[:, :, i] - sub[:, i, None] * rp[-1]) / den[:, None])
    mm = [rp[-1]]
    for i in range(n - 2, -1, -1):
        mm.append(rp[i] - cp[i][:, None] * mm[-1])
    mm.reverse()
    M = torch.stack(mm, dim=-1)
    first = ((h[:, 0] + h[:, 1])[:, None] * M[:, :, 0] - h[:, 0, None] * M[:, :, 1]) / h[:, 1, None]
    last = ((h[:, -1] + h[:, -2])[:, None] * M[:, :, -1] - h[:, -1, None] * M[:, :, -2]) / h[:, -2, None]
    M = torch.cat([first[..., None], M, last[..., None]], dim=-1)
    hh = h[:, None]
    return torch.stack([y[:, :, :-1], sl - hh * (2 * M[:, :, :-1] + M[:, :, 1:]) / 6, 0.5 * M[:, :, :-1],
                        (M[:, :, 1:] - M[:, :, :-1]) / (6 * hh)])


def _turns(f, tc):
    """f tc modulo 1, with the product's rounding error put back (Dekker's product)."""
    big = 134217729.0
    c = big * f
    fh = c - (c - f)
    fl = f - fh
    d = big * tc
    th = d - (d - tc)
    tl = tc - th
    p = f * tc
    return (p - torch.round(p)) + (((fh * th - p) + fh * tl + fl * th) + fl * tl)


class _Template:
    """Splined templates of parameter rows th on the grid, one walker's modes at a time."""

    def __init__(self, th, modes, K, f0, df, n, t0):
        self.s = _source(np.asarray(th), t0)
        self.tc = self.s["tc"].cpu().numpy()
        sc = _col(self.s)
        k = torch.arange(K, dtype=torch.float64, device=_dev()) / (K - 1)
        self.f0, self.df, self.K, self.parts = f0, df, K, []
        for l, m in modes:
            act, lo, hi, jl, jh = _bands(self.s, m, f0, df, n)
            good = torch.as_tensor(act, device=_dev())[:, None]
            lo = torch.where(good, lo[:, None], torch.full_like(lo[:, None], 1e-3))
            hi = torch.where(good, hi[:, None], torch.full_like(hi[:, None], 2e-3))
            f = lo * torch.exp(torch.log(hi / lo) * k)
            f[:, -1:] = hi
            a, p = _amp_phase(sc, l, m, f)
            T, delay = _response(sc, l, m, f)
            y = torch.stack([a, p + delay] + [g for c in range(3) for g in (T[c].real, T[c].imag)], dim=1)
            self.parts.append((act, jl, jh, f, _spline(f, y)))

    def modes_of(self, w):
        """(first bin, h [3, bins, 2] or None) of every mode of walker w."""
        for act, jl, jh, fk, coef in self.parts:
            if not act[w]:
                yield 0, None
                continue
            a, b = int(jl[w]), int(jh[w])
            f = self.f0 + torch.arange(a, b + 1, dtype=torch.float64, device=_dev()) * self.df
            seg = (torch.searchsorted(fk[w], f, right=True) - 1).clamp(0, self.K - 2)
            x = f - fk[w][seg]
            c = coef[:, w].permute(2, 0, 1).reshape(self.K - 1, 32)[seg]  # [bins, 32]
            c = c.reshape(-1, 4, 8)
            v = c[:, 0] + x[:, None] * (c[:, 1] + x[:, None] * (c[:, 2] + x[:, None] * c[:, 3]))
            ph = v[:, 1] - TWO_PI * _turns(f, float(self.tc[w]))
            zr, zi = v[:, 0] * torch.cos(ph), v[:, 0] * torch.sin(ph)
            h = torch.empty((3, f.shape[0], 2), dtype=torch.float64, device=_dev())
            for ch in range(3):
                tr, ti = v[:, 2 + 2 * ch], v[:, 3 + 2 * ch]
                h[ch, :, 0] = tr * zr - ti * zi
                h[ch, :, 1] = tr * zi + ti * zr
            yield a, h


def _exact_loglike(case, seed):
    f0, df, n, t0, d, psd = _data(case, seed)
    th = _walkers(case, seed)
    B = th.shape[0]
    w = 4 * df / psd
    wd = w[:, :, None] * d
    dd = float((wd * d).sum())
    out = np.zeros((3, B))
    group = 256
    for b0 in range(0, B, group):
        tm = _Template(th[b0:b0 + group], MODES[:case["modes"]], case["knots"], f0, df, n, t0)
        for i in range(len(tm.tc)):
            if not tm.s["ok"][i]:
                out[:, b0 + i] = (-np.inf, 0.0, 0.0)
                continue
            ms = [(j, h) for j, h in tm.modes_of(i) if h is not None]
            dh = hh = 0.0
            if ms:
                lo, hi = min(j for j, _ in ms), max(j + h.shape[1] for j, h in ms)
                tot = torch.zeros((3, hi - lo, 2), dtype=torch.float64, device=_dev())
                for j, h in ms:
                    tot[:, j - lo:j - lo + h.shape[1]] += h
                dh = float((wd[:, lo:hi] * tot).sum())
                hh = float((w[:, lo:hi, None] * tot * tot).sum())
            out[:, b0 + i] = (dh - 0.5 * hh - 0.5 * dd, dh, hh)
    if case["api"] == "host":
        return out[0], out[1], out[2]
    return _t(out[0]) if case["precision"] == "split" else (_t(out[0]), _t(out[1]), _t(out[2]))


def _exact_cross(case, seed):
    f0, df, n, t0 = _grid(case)
    w = 4 * df / _psd(_freqs(f0, df, n))
    th = _walkers(case, seed)
    L = case["modes"]
    tm = _Template(th, MODES[:L], case["knots"], f0, df, n, t0)
    out = np.zeros((th.shape[0], L, L))
    for b in range(th.shape[0]):
        ms = list(tm.modes_of(b))
        for i in range(L):
            for k in range(i, L):
                (ja, ha), (jb, hb) = ms[i], ms[k]
                if ha is None or hb is None:
                    continue
                lo, hi = max(ja, jb), min(ja + ha.shape[1], jb + hb.shape[1])
                if lo < hi:
                    x = ha[:, lo - ja:hi - ja] * hb[:, lo - jb:hi - jb] * w[:, lo:hi, None]
                    out[b, i, k] = out[b, k, i] = float(x.sum())
    return out


def _direct(s, l, m, f, band):
    """The mode's A, E, T template at the frequencies themselves, [3, B, F] complex."""
    a, p = _amp_phase(s, l, m, f)
    T, delay = _response(s, l, m, f)
    z = torch.polar(torch.ones_like(a), p + delay - TWO_PI * _turns(f, s["tc"]))
    return torch.where(band, a * T * z, torch.zeros_like(a * T))


def _exact_rb(case, seed):
    f0, df, n, t0, d, psd = _data(case, seed)
    w = 4 * df / psd
    dc = torch.view_as_complex(d.contiguous())
    dd = float((w * (dc.real ** 2 + dc.imag ** 2)).sum())
    modes = MODES[:case["modes"]]
    fid = _source(_injection(case)[None, :], t0)
    bands = [_bands(fid, m, f0, df, n) for _, m in modes]
    ed = [j for b in bands if b[0][0] for j in (int(b[3][0]), int(b[4][0]) + 1)]
    lo, hi = min(ed), max(ed)
    fl, fh = f0 + lo * df, f0 + hi * df
    step = (math.log(fh) - math.log(fl)) / case["bins"]
    ys = [math.log(fl) + i * step for i in range(case["bins"])] + [math.log(fh)]
    ed += [int(min(max(np.rint((math.exp(y) - f0) / df), lo), hi)) for y in ys]
    ed = np.unique(np.array(ed, dtype=np.int64))
    nb = len(ed) - 1
    e = torch.as_tensor(ed, device=_dev())
    fe = f0 + e.to(torch.float64) * df
    j = torch.arange(lo, hi, device=_dev())
    f = f0 + j.to(torch.float64) * df
    b = (torch.searchsorted(e, j, right=True) - 1).clamp(0, nb - 1)
    x1 = f - fe[b]
    sc = _col(fid)

    def inside(q, ff):
        return (ff >= q[1][:, None]) & (ff <= q[2][:, None]) & torch.as_tensor(q[0], device=_dev())[:, None]

    h0 = [_direct(sc, l, m, f[None], inside(q, f[None]))[:, 0] for (l, m), q in zip(modes, bands)]
    h0e = [_direct(sc, l, m, fe[None], inside(q, fe[None]))[:, 0] for (l, m), q in zip(modes, bands)]

    def per_bin(v):  # [3, bins] complex -> sums over coarse bins
        o = torch.zeros((3, nb, 2), dtype=torch.float64, device=_dev())
        return torch.view_as_complex(o.index_add_(1, b, torch.view_as_real(v.contiguous())))

    ww, wd = w[:, lo:hi], (w * dc)[:, lo:hi]
    th = _walkers(case, seed)
    src = _source(th, t0)
    sw = _col(src)
    r0, r1 = [], []
    for (l, m), g in zip(modes, h0e):
        h = _direct(sw, l, m, fe[None], inside(_bands(src, m, f0, df, n), fe[None]))  # [3, B, ne]
        ok = (g != 0)[:, None, :]
        r = torch.where(ok, h / torch.where(ok, g[:, None, :], torch.ones_like(g[:, None, :])),
                        torch.zeros_like(h))
        okl, okr, rl, rr = ok[..., :-1], ok[..., 1:], r[..., :-1], r[..., 1:]
        r0.append(torch.where(okl, rl, torch.where(okr, rr, torch.zeros_like(rl))))
        r1.append(torch.where(okl & okr, (rr - rl) / (fe[1:] - fe[:-1]), torch.zeros_like(rl)))
    dh = torch.zeros(th.shape[0], dtype=torch.float64, device=_dev())
    hh = torch.zeros_like(dh)
    for a in range(len(modes)):
        v = wd * h0[a].conj()
        A0, A1 = per_bin(v), per_bin(v * x1)
        dh += (A0[:, None] * r0[a].conj() + A1[:, None] * r1[a].conj()).real.sum(dim=(0, 2))
        for c in range(a, len(modes)):
            v = ww * h0[a] * h0[c].conj()
            B0, B1 = per_bin(v), per_bin(v * x1)
            t = B0[:, None] * r0[a] * r0[c].conj() + B1[:, None] * (r0[a] * r1[c].conj() + r1[a] * r0[c].conj())
            hh += (1.0 if a == c else 2.0) * t.real.sum(dim=(0, 2))
    return dh - 0.5 * hh - 0.5 * dd, dh, hh


def _kept(c):
    d = torch.arange(FLOW_D, device=_dev())
    return [(d % 2 == 0), (d % 2 == 1), (d < 6), (d >= 6)][c % 4]


def _coupling(w, c, u):
    k = _kept(c)
    a = torch.relu(torch.where(k, u, torch.zeros_like(u)) @ w["W1"][c].T + w["b1"][c])
    o = torch.relu(a @ w["W2"][c].T + w["b2"][c]) @ w["W3"][c].T + w["b3"][c]
    zero = torch.zeros_like(u)
    return (torch.where(k, zero, 2.0 * torch.tanh(o[:, :FLOW_D] / 2.0)),
            torch.where(k, zero, o[:, FLOW_D:]))


def _to_z(w, u):
    tot = 0.0
    for c in range(FLOW_C):
        s, t = _coupling(w, c, u)
        u = (u - t) * torch.exp(-s)
        tot = tot + s.sum(dim=1)
    return u, tot


def _exact_flow(case, seed):
    n = case["rows"]
    w = {k: _t(v) for k, v in _flow_weights(seed).items()}
    mu, L = (_t(a) for a in _whitening(_chain(seed + 1, 4000)))
    norm = 0.5 * FLOW_D * math.log(TWO_PI) + torch.log(torch.diagonal(L)).sum()
    z = _t(np.random.default_rng([seed, 21]).standard_normal((n, 11)))
    u, tot = z, 0.0
    for c in reversed(range(FLOW_C)):
        s, t = _coupling(w, c, u)
        u = u * torch.exp(s) + t
        tot = tot + s.sum(dim=1)
    y, qy = mu + u @ L.T, -0.5 * (z * z).sum(dim=1) - norm - tot
    x = _t(_chain(seed, n + 64)[:n])
    v, tot = _to_z(w, torch.linalg.solve_triangular(L, (x - mu).T, upper=False).T)
    return {"y": y, "qy": qy, "u": v, "qx": -0.5 * (v * v).sum(dim=1) - norm - tot}


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on uint64 arrays that hold 32-bit words; four arrays."""
    m = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = ((p1 >> np.uint64(32)) ^ c1 ^ k0) & m, p1 & m, ((p0 >> np.uint64(32)) ^ c3 ^ k1) & m, p0 & m
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m, (k1 + np.uint64(0xBB67AE85)) & m
    return c0, c1, c2, c3


def _exact_train(case, seed):
    x = _chain(seed, case["rows"] + 64)[:case["rows"]]
    mu, L = _whitening(x)
    U = torch.linalg.solve_triangular(_t(L), (_t(x) - _t(mu)).T, upper=False).T.contiguous()
    w = {k: _t(v).requires_grad_(True) for k, v in _flow_weights(seed).items()}
    m1 = {k: torch.zeros_like(v) for k, v in w.items()}
    m2 = {k: torch.zeros_like(v) for k, v in w.items()}
    loss = np.empty(case["iters"])
    j = np.arange(case["batch"], dtype=np.uint64)
    for it in range(case["iters"]):
        z64 = np.zeros_like(j)
        q = np.stack(_philox(z64, z64 + np.uint64(5), z64 + np.uint64(it), j >> np.uint64(2),
                             z64 + np.uint64(1), z64))
        r = (q[(j & np.uint64(3)).astype(int), np.arange(len(j))].astype(np.float64) + 0.5) * 2.0 ** -32
        rows = np.minimum((r * case["rows"]).astype(np.int64), case["rows"] - 1)
        z, tot = _to_z(w, U[torch.as_tensor(rows, device=_dev())])
        val = (0.5 * (z * z).sum(dim=1) + tot).mean()
        loss[it] = float(val.detach())
        g = dict(zip(w, torch.autograd.grad(val, list(w.values()))))
        with torch.no_grad():
            for k in w:
                m1[k] = 0.9 * m1[k] + 0.1 * g[k]
                m2[k] = 0.999 * m2[k] + 0.001 * g[k] ** 2
                w[k] -= 1e-3 * (m1[k] / (1 - 0.9 ** (it + 1))) / (torch.sqrt(m2[k] / (1 - 0.999 ** (it + 1))) + 1e-8)
    return {"loss": loss, "weights": {k: v.detach().cpu().numpy() for k, v in w.items()}}


def exact(case, seed):
    kind = case["kind"]
    if kind == "loglike":
        mb, _, _ = _active_bins(case)
        return None if mb > 2e10 else _exact_loglike(case, seed)  # beyond: too long
    return {"rb": _exact_rb, "cross": _exact_cross, "flow": _exact_flow, "train": _exact_train,
            "sampler": lambda c, s: None}[kind](case, seed)  # a chain is a sequence of decisions
