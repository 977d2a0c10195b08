"""Timed cases of the transit search: the calls a survey program makes.

Each case is one call (or one short chain of calls) of the public binding on
synthetic TESS-shaped light curves: 2-minute cadence, one to seven sectors,
gaps, dropped cadences, times at the spacecraft (a regular grid) or corrected
to the barycentre (the light-travel term makes the spacing drift, so the grid
is not regular), FP64 and mixed precision.

kinds
  chain    nu_gp_factor + nu_linear_search + nu_periodic_search
  events   nu_gp_factor + nu_linear_search
  linear   nu_linear_search on a factor that is already held
  fold     nu_periodic_search on a grid of single events
  refine   nu_periodic_refine of candidates on a factor that is already held
  batch    nu_batch_search of a survey of curves of uneven length
"""
import math
import random

import numpy as np
import torch

from paper_2402_06835_gb300 import api, synth

CADENCE = 2.0 / 1440.0
SIZE_SEED = 20240206


# ------------------------------------------------------------------ the cases
def listed():
    return [
        dict(name="chain_2048_5d_fp64", kind="chain", n=2048, n_d=5, d_lo=0.5, d_hi=2.0,
             n_p=1000, p_lo=0.3, p_hi=1.4, grid="linear", precision="fp64",
             template="box", terms="rotation", k=2, gaps=0, drop=0.0, bary=False),
        dict(name="events_19440_16d_mixed", kind="events", n=19440, n_d=16, d_lo=1.0 / 3,
             d_hi=3.0, precision="mixed", template="box", terms="rotation", k=2, gaps=1,
             drop=0.0, bary=False),
        dict(name="events_136080_20d_fp64", kind="events", n=136080, n_d=20, d_lo=0.25,
             d_hi=4.0, precision="fp64", template="box", terms="rotation", k=2, gaps=13,
             drop=0.0, bary=False),
        dict(name="linear_19440_10d_trapezoid_fp64", kind="linear", n=19440, n_d=10,
             d_lo=1.0 / 3, d_hi=3.0, precision="fp64", template="trapezoid",
             terms="rotation", k=2, gaps=1, drop=0.01, bary=True),
        dict(name="fold_19440_10d_fp64", kind="fold", n=19440, n_d=10, d_lo=1.0 / 3, d_hi=3.0,
             n_p=20000, p_lo=0.2, p_hi=13.5, grid="linear", precision="fp64", gaps=1,
             drop=0.0, bary=False, masked=False),
        dict(name="fold_19440_16d_mixed", kind="fold", n=19440, n_d=16, d_lo=1.0 / 3, d_hi=3.0,
             n_p=20000, p_lo=0.2, p_hi=13.5, grid="linear", precision="mixed", gaps=1,
             drop=0.0, bary=False, masked=False),
        dict(name="fold_bary_19440_10d_fp64", kind="fold", n=19440, n_d=10, d_lo=1.0 / 3,
             d_hi=3.0, n_p=20000, p_lo=0.2, p_hi=13.5, grid="linear", precision="fp64",
             gaps=1, drop=0.01, bary=True, masked=False),
        dict(name="fold_bary_19440_10d_mixed", kind="fold", n=19440, n_d=10, d_lo=1.0 / 3,
             d_hi=3.0, n_p=20000, p_lo=0.2, p_hi=13.5, grid="linear", precision="mixed",
             gaps=1, drop=0.01, bary=True, masked=True),
        dict(name="fold_136080_20d_mixed", kind="fold", n=136080, n_d=20, d_lo=0.25, d_hi=4.0,
             n_p=100000, p_lo=0.2, p_hi=50.0, grid="linear", precision="mixed", gaps=13,
             drop=0.0, bary=False, masked=False),
        dict(name="refine_19440_64", kind="refine", n=19440, n_d=10, d_lo=1.0 / 3, d_hi=3.0,
             n_c=64, p_lo=0.2, p_hi=13.5, template="box", terms="rotation", k=2, gaps=1,
             drop=0.0, bary=False),
        dict(name="batch_survey_438_mixed", kind="batch", n_lc=438, n_lo=8000, n_hi=20000,
             n_d=10, d_lo=1.0 / 3, d_hi=3.0, n_p=4000, p_lo=0.3, p_hi=10.0, grid="linear",
             precision="mixed", terms="rotation", k=2, gaps=2),
        dict(name="batch_injection_1000_fp64", kind="batch", n_lc=1000, n_lo=2880, n_hi=2880,
             n_d=1, d_lo=0.96, d_hi=0.96, n_p=4000, p_lo=0.3, p_hi=3.0, grid="linear",
             precision="fp64", terms="sho", k=2, gaps=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# most events (period x sample x duration) of a drawn fold: those of the listed
# ones, less where every event costs more (small share of regular cells pruned)
_MAX_EVENTS = 3.8e9


def draw(rng):
    kind = rng.choices(["chain", "events", "linear", "fold", "refine", "batch"],
                       [2, 2, 3, 7, 1, 3])[0]
    d_lo = rng.uniform(0.25, 1.0)
    d_hi = d_lo * rng.uniform(1.5, 8.0)
    case = dict(kind=kind, d_lo=d_lo, d_hi=d_hi)
    terms = rng.choice(["rotation", "rotation", "sho", "rotation+sho", "rotation+exp"])
    precision = rng.choice(["fp64", "mixed"])
    irregular = dict(gaps=rng.randint(0, 4), drop=rng.choice([0.0, 0.0, 0.01, 0.03]),
                     bary=rng.random() < 0.5)
    if kind == "batch":
        n_hi = _log_int(rng, 1500, 20000)
        n_lo = int(n_hi * rng.uniform(0.4, 1.0))
        n_d = rng.randint(1, 12)
        n_lc = _log_int(rng, 8, 438)
        n_p = _log_int(rng, 300, 4000)
        n_p = max(200, min(n_p, int(3.0e10 / (n_lc * n_hi * n_d))))
        span = n_lo * CADENCE
        case.update(n_lc=n_lc, n_lo=n_lo, n_hi=n_hi, n_d=n_d, n_p=n_p, p_lo=0.3,
                    p_hi=max(0.6, rng.uniform(0.3, 0.7) * span),
                    grid=rng.choice(["linear", "frequency"]), precision=precision,
                    terms=rng.choice(["rotation", "sho"]), k=rng.choice([1, 2]),
                    gaps=rng.randint(0, 2))
        return case
    if kind == "refine":
        n = _log_int(rng, 2000, 30000)
        case.update(n=n, n_d=rng.randint(1, 16), n_c=_log_int(rng, 1, 256), p_lo=0.3,
                    p_hi=max(0.6, 0.5 * n * CADENCE), template=rng.choice(["box", "trapezoid"]),
                    terms=terms, k=rng.choice([1, 2, 3]), **irregular)
        return case
    n_hi = {"chain": 30000, "events": 136080, "linear": 136080, "fold": 136080}[kind]
    n = _log_int(rng, 1024, n_hi)
    n_d = rng.randint(1, 20)
    if kind in ("chain", "fold"):
        n_p = _log_int(rng, 300, 30000)
        n_p = max(100, min(n_p, int(_MAX_EVENTS / (n * n_d))))
        case.update(n_p=n_p, p_lo=rng.uniform(0.2, 0.5),
                    p_hi=max(0.7, rng.uniform(0.3, 0.6) * n * CADENCE),
                    grid=rng.choice(["linear", "frequency"]))
    if kind == "fold":
        case.update(n=n, n_d=n_d, precision=precision, masked=rng.random() < 0.3, **irregular)
        return case
    template = rng.choice(["box", "box", "box", "trapezoid", "limb_quad"])
    case.update(n=n, n_d=n_d, precision=precision, template=template, terms=terms,
                k=rng.choice([0, 1, 2, 2, 3]), **irregular)
    return case


# ------------------------------------------------------------------- inputs
def _sizes(case):
    """Sample counts of a batch's curves (fixed by the case, not by the seed)."""
    r = random.Random(SIZE_SEED + case["n_lc"])
    return [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case["n_lc"])]


def _slots(n, gaps, drop, rng):
    """Slots of n samples on the 2-minute grid: evenly spaced data gaps of a day
    or less, and a fraction of single dropped cadences."""
    gap = min(720, max(8, n // 20))
    extra = int(rng.binomial(n, drop)) if drop > 0 else 0
    total = n + extra
    idx = np.arange(total) + (np.arange(total) * (gaps + 1) // total) * gap
    if extra:
        idx = np.delete(idx, 1 + rng.choice(total - 2, extra, replace=False))
    return idx


def _times(slots, bary, rng):
    """Sample times; with bary, at the solar-system barycentre (light-travel
    term of a 1-au orbit, 499 s times the cosine of the ecliptic latitude)."""
    if not bary:
        return slots * CADENCE
    t = 1325.0 + slots * CADENCE
    amp = 499.0 / 86400.0 * rng.uniform(0.3, 1.0)
    return t + amp * np.sin(2.0 * np.pi * t / 365.25 + rng.uniform(0.0, 2.0 * np.pi))


def _durations(case):
    return np.linspace(case["d_lo"], case["d_hi"], case["n_d"]) / 24.0


def _periods(case):
    if case["grid"] == "frequency":
        return 1.0 / np.linspace(1.0 / case["p_lo"], 1.0 / case["p_hi"], case["n_p"])
    return np.linspace(case["p_lo"], case["p_hi"], case["n_p"])


def _terms(name, sigma, p_rot):
    rot = (synth.TERM_ROTATION, (sigma, p_rot, 5.0, 0.0, 0.5))
    sho = (synth.TERM_SHO, (0.3 * sigma, 2.0 * np.pi / (2.5 * p_rot), 0.7, 0.0, 0.0))
    exp = (synth.TERM_EXP, (0.3 * sigma, 3.0 * p_rot, 0.0, 0.0, 0.0))
    return {"rotation": [rot], "rotation+sho": [rot, sho], "rotation+exp": [rot, exp],
            "sho": [(synth.TERM_SHO, (sigma, 2.0 * np.pi / p_rot, 5.0, 0.0, 0.0))]}[name]


def _design(t, k):
    x = (t - t[0]) / (t[-1] - t[0])
    return np.stack([np.ones_like(t), x, x * x][:k], axis=1) if k else np.zeros((len(t), 0))


def _curve(case, seed):
    """One light curve with rotation-like variability and an injected transit."""
    rng = np.random.default_rng([seed, case["n"]])
    slots = _slots(case["n"], case["gaps"], case["drop"], rng)
    span = (slots[-1] + 1) * CADENCE
    p_rot = 1.2 if span > 8.0 else 0.5
    inject = (1.5e-3, 1.5 / 24.0, min(3.1, span / 4.0))
    lc = synth.make_curve(rng, slots, 0.0, p_rot, 2e-2, 2e-3, inject=inject, design=False)
    t = _times(slots, case["bary"], rng)
    return dict(t=t, y=lc.y, dv=lc.diag_var, terms=_terms(case["terms"], 2e-2, p_rot),
                X=_design(t, case["k"]), inject=dict(lc.injected, epoch=lc.injected["epoch"]
                                                     - lc.t[0] + t[0]))


def _events(case, seed):
    """Single events (depth, var, gain) of a light curve whose variability has
    been modelled: box depths against the window's shoulders in white noise
    with an injected planet; with masked, a second planet's transits removed
    from the grid (NaN), as a multi-planet search leaves them."""
    rng = np.random.default_rng([seed, case["n"]])
    slots = _slots(case["n"], case["gaps"], case["drop"], rng)
    t = _times(slots, case["bary"], rng)
    span = t[-1] - t[0]
    sw = 2e-3
    y = sw * rng.standard_normal(len(t))
    period = min(3.1, span / 4.0) * rng.uniform(0.9, 1.1)
    y[np.abs((t - t[0] - rng.uniform(0, period) + 0.5 * period) % period - 0.5 * period)
      < 0.75 / 24.0] -= 1.5e-3
    cs = np.concatenate([[0.0], np.cumsum(y)])
    depth, var = [], []
    for D in _durations(case):
        lo, hi = np.searchsorted(t, t - D * 0.5), np.searchsorted(t, t + D * 0.5)
        a, b = np.searchsorted(t, t - D), np.searchsorted(t, t + D)
        n_in = np.maximum(hi - lo, 1)
        n_out = (lo - a) + (b - hi)
        s_out = (cs[lo] - cs[a]) + (cs[b] - cs[hi])
        base = np.where(n_out > 0, s_out / np.maximum(n_out, 1), 0.0)
        d = base - (cs[hi] - cs[lo]) / n_in
        v = sw * sw * (1.0 / n_in + np.where(n_out > 0, 1.0 / np.maximum(n_out, 1), 0.0))
        empty = hi <= lo
        depth.append(np.where(empty, np.nan, d))
        var.append(np.where(empty, np.nan, v))
    depth, var = np.stack(depth), np.stack(var)
    if case["masked"]:
        p2 = 0.37 * period + 0.2
        gone = np.abs((t - t[0]) % p2 - 0.5 * p2) < 1.5 / 24.0
        depth[:, gone] = np.nan
        var[:, gone] = np.nan
    ft = np.float32 if case["precision"] == "mixed" else np.float64
    depth, var = depth.astype(ft), var.astype(ft)
    return t, depth, var, depth * depth / (2 * var)


def _batch(case, seed):
    """Curves of a survey: uneven lengths, gaps, a planet in every second one."""
    curves = []
    for c, n in enumerate(_sizes(case)):
        rng = np.random.default_rng([seed, c, n])
        slots = _slots(n, case["gaps"], 0.0, rng)
        p_rot = float(np.exp(rng.uniform(np.log(0.1), np.log(5.0))))
        sigma = float(np.exp(rng.uniform(np.log(1e-3), np.log(5e-2))))
        inject = None
        if c % 2 == 0:
            inject = (float(np.exp(rng.uniform(np.log(5e-4), np.log(1e-2)))),
                      float(rng.uniform(0.5, 3.0)) / 24.0,
                      float(rng.uniform(0.5, max(1.0, 0.3 * n * CADENCE))))
        lc = synth.make_curve(rng, slots, 0.0, p_rot, sigma, float(rng.uniform(1e-3, 5e-3)),
                              inject=inject, design=False)
        curves.append((lc.t, lc.y, lc.diag_var, _terms(case["terms"], sigma, p_rot)))
    return curves


def _candidates(case, seed, t, inject):
    """Candidates as a search's best periods give them: the injected period,
    its aliases and their neighbours, and unrelated ones."""
    rng = np.random.default_rng([seed, 7])
    Ds = _durations(case)
    P, T0, idx = [], [], []
    for i in range(case["n_c"]):
        if i % 2 == 0:
            p = inject["period"] * [1.0, 2.0, 0.5, 3.0, 1.0 / 3.0][(i // 2) % 5]
            p *= 1.0 + 1e-3 * rng.standard_normal() * (i > 8)
        else:
            p = rng.uniform(case["p_lo"], case["p_hi"])
        fits = np.nonzero(2.0 * Ds <= p)[0]
        P.append(p)
        T0.append(t[0] + rng.uniform(0.0, p))
        idx.append(int(rng.choice(fits)) if len(fits) else 0)
    return np.array(P), np.array(T0), np.array(idx, dtype=np.int32)


def _cu(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _factor(s):
    return api.nu_gp_factor(s["t"], s["dv"], s["terms"], s["X"], s["y"])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, Ds=_durations(case), precision=case.get("precision", "fp64"),
             template=case.get("template", "box"))
    if kind == "batch":
        s["curves"] = [(_cu(t), _cu(y), _cu(dv), terms)
                       for t, y, dv, terms in _batch(case, seed)]
        s["periods"] = _cu(_periods(case))
        s["k"] = case["k"]
        return s
    if kind == "fold":
        s["t"], s["depth"], s["var"], s["dlnl"] = (_cu(a) for a in _events(case, seed))
        s["periods"] = _cu(_periods(case))
        return s
    lc = _curve(case, seed)
    s.update(t=_cu(lc["t"]), y=_cu(lc["y"]), dv=_cu(lc["dv"]), X=_cu(lc["X"]),
             terms=lc["terms"])
    if kind == "chain":
        s["periods"] = _cu(_periods(case))
    if kind == "refine":
        s["P"], s["T0"], s["idx"] = (_cu(a) for a in
                                     _candidates(case, seed, lc["t"], lc["inject"]))
    if kind in ("linear", "refine"):
        s["factor"] = _factor(s)
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        out = api.nu_batch_search(s["curves"], s["Ds"], s["periods"], k=s["k"],
                                  precision=s["precision"])
        return dict(out, status=np.asarray(out["status"], dtype=np.int32))
    if kind == "fold":
        return api.nu_periodic_search(s["t"], s["Ds"], s["depth"], s["var"], s["dlnl"],
                                      s["periods"], precision=s["precision"])
    if kind == "refine":
        return api.nu_periodic_refine(s["factor"], s["P"], s["T0"], s["idx"], s["Ds"],
                                      template=s["template"])
    f = s["factor"] if kind == "linear" else _factor(s)
    depth, var, dlnl = api.nu_linear_search(f, s["t"], s["Ds"], template=s["template"],
                                            precision=s["precision"])
    out = dict(depth=depth, var=var, dlnl=dlnl)
    if kind == "chain":
        out["periodic"] = api.nu_periodic_search(s["t"], s["Ds"], depth, var, dlnl,
                                                 s["periods"], precision=s["precision"])
    return out


# ----------------------------------------------------------- necessary work
_J = {"rotation": 4, "sho": 2, "rotation+sho": 6, "rotation+exp": 6}


def work(case):
    """Inputs read once and outputs written once; operations of the O(N)
    algorithms: the factor's recursions, one window recursion per start
    epoch, one addition per (cell, event) of a fold."""
    kind = case["kind"]
    el = 4 if case.get("precision") == "mixed" else 8
    n_d = case["n_d"]
    ns = _sizes(case) if kind == "batch" else [case["n"]]
    n = sum(ns)
    by = fl = 0
    if kind != "fold":
        J, k = _J[case["terms"]], case["k"]
        if kind in ("chain", "events", "batch"):
            by += 8 * n * (3 + (k if kind != "batch" else 0))
            fl += n * (6 * J * J + 8 * J * (k + 1))
        else:
            # the held factor: transitions, gain, pivot, future information, residual, X
            by += 8 * n * (1 + 2 * J + J + 1 + J * (J + 1) // 2 + 1 + k)
    if kind in ("chain", "events", "linear", "batch"):
        length = _durations(case) / CADENCE
        steps = length.max() if case.get("template", "box") == "box" else length.sum()
        fl += int(n * (steps * (8 + 6 * J) + n_d * (J * J + 2 * J + 4 * k + 8)))
        if kind in ("events", "linear", "chain"):
            by += 3 * n_d * n * el
    if kind == "refine":
        by += case["n_c"] * (8 + 8 + 4 + 32)
        fl += int(case["n_c"] * n * 2 * J)
    if kind in ("chain", "fold", "batch"):
        n_p = case["n_p"]
        if kind == "fold":
            by += 8 * n + 3 * n_d * n * el
        by += 8 * n_p + 44 * n_p * len(ns)
        fl += n * n_d * n_p
    return {"bytes": int(by), "flops": int(fl)}


# ------------------------------------------- the same outputs in plain FP64
def _covariance(t, dv, terms):
    tau = (t[:, None] - t[None, :]).abs_()
    S = torch.zeros_like(tau)

    def sho(sigma, omega, Q):
        x = tau * (omega / (2.0 * Q))
        f = math.sqrt(abs(4.0 * Q * Q - 1.0))
        S.add_(torch.exp(-x).mul_(torch.cos(f * x) + torch.sin(f * x) / f), alpha=sigma ** 2)

    for kind, p in terms:
        if kind == synth.TERM_SHO:
            sho(*p[:3])
        elif kind == synth.TERM_EXP:
            S.add_(torch.exp(-tau / p[1]), alpha=p[0] ** 2)
        else:
            sigma, period, q0, dq, f = p
            q1, q2 = 0.5 + q0 + dq, 0.5 + q0
            w1 = 4.0 * math.pi * q1 / (period * math.sqrt(4.0 * q1 * q1 - 1.0))
            sho(sigma / math.sqrt(1.0 + f), w1, q1)
            sho(sigma * math.sqrt(f / (1.0 + f)), 2.0 * w1, q2)
    S.diagonal().add_(dv)
    return S


def _template(kind, t, t0, D):
    """Unit-depth template (positive) of samples t about epochs t0."""
    inside = (t >= t0 - D * 0.5) & (t < t0 + D * 0.5)
    if kind == "box":
        m = torch.ones_like(t)
    elif kind == "trapezoid":
        m = ((D * 0.5 - (t - t0).abs()) / (0.1 * D)).clamp(0.0, 1.0)
    else:
        r = torch.where(inside, 2.0 * (t - t0) / D, torch.zeros_like(t))
        x = 1.0 - torch.sqrt(1.0 - r * r)
        m = 1.0 - 0.4 * x - 0.25 * x * x
    return torch.where(inside, -m, torch.zeros_like(m))


def _dense(lc):
    """Cholesky factor of the covariance, Sigma^-1 r0 and Sigma^-1 X R^-1."""
    t, y, dv, X = (_cu(lc[a]) for a in ("t", "y", "dv", "X"))
    C = torch.linalg.cholesky(_covariance(t, dv, lc["terms"]))
    yw = torch.linalg.solve_triangular(C, y[:, None], upper=False)
    Q = torch.linalg.qr(torch.linalg.solve_triangular(C, X, upper=False))[0]
    r = yw - Q @ (Q.T @ yw)
    Z = torch.linalg.solve_triangular(C.T, torch.cat([r, Q], dim=1), upper=True)
    return t, C, Z[:, 0].contiguous(), Z[:, 1:].contiguous()


def _finish(c, num, b):
    s = c - (b * b).sum(-1)
    nan = torch.full_like(c, math.nan)
    ok = c > 0
    return (torch.where(ok, num / s, nan), torch.where(ok, 1.0 / s, nan),
            torch.where(ok, num * num / (2.0 * s), nan))


def _exact_linear(case, lc):
    t, C, z0, Z = _dense(lc)
    n = len(t)
    S = torch.cholesky_inverse(C)
    del C
    Sf = S.reshape(-1)
    out = []
    for D in _durations(case):
        lo = torch.searchsorted(t, t - D * 0.5)
        L = int((torch.searchsorted(t, t + D * 0.5) - lo).max())
        idx = (lo[:, None] + torch.arange(L, device="cuda")[None]).clamp_(max=n - 1)
        m = _template(case["template"], t[idx], t[:, None], D)
        # past the last sample the clamped index would repeat it
        m = torch.where(lo[:, None] + torch.arange(L, device="cuda")[None] < n, m,
                        torch.zeros_like(m))
        c = torch.zeros_like(t)
        for a in range(L):
            row = Sf[idx[:, a:a + 1] * n + idx]
            c += m[:, a] * (row * m).sum(1)
        num = (z0[idx] * m).sum(1)
        b = torch.stack([(Z[:, i][idx] * m).sum(1) for i in range(Z.shape[1])], dim=1) \
            if Z.shape[1] else torch.zeros((n, 0), dtype=t.dtype, device="cuda")
        out.append(_finish(c, num, b))
    return [torch.stack([o[i] for o in out]) for i in range(3)]


def _exact_fold(case, t, depth, var, dlnl):
    depth, var, dlnl = depth.double(), var.double(), dlnl.double()
    n = len(t)
    diff = t[1:] - t[:-1]
    dt = float(np.median(diff.cpu().numpy()))
    sig = torch.sqrt(torch.where(var > 0, var, torch.full_like(var, math.nan)))
    node = torch.isfinite(depth) & torch.isfinite(sig) & torch.isfinite(dlnl)
    pair = node[:, :-1] & node[:, 1:] & (diff <= 1.5 * dt)[None]
    t_ref, t_last = t[0].item(), t[-1].item()
    n_d = depth.shape[0]
    vals = torch.stack([depth, sig, dlnl])
    vals = torch.where(node[None], vals, torch.zeros_like(vals))
    zero = torch.zeros((), dtype=t.dtype, device="cuda")
    best = []
    for P in _periods(case).tolist():
        n_phi = math.ceil(P / dt)
        k_max = int(math.floor((t_last - t_ref) / P)) + 2
        phi = torch.arange(n_phi, dtype=t.dtype, device="cuda") / n_phi
        T = t_ref + (phi[:, None] + torch.arange(k_max, dtype=t.dtype, device="cuda")) * P
        i = (torch.searchsorted(t, T, right=True) - 1).clamp_(max=n - 2)
        ta = t[i]
        w = (T - ta) / diff[i]
        valid = pair[:, i] & ((T <= t_last) & (T < t[-1]))[None]
        va, vb = vals[:, :, i], vals[:, :, i + 1]
        d_k, s_k, l_k = (1.0 - w) * va + w * vb
        sk2 = s_k * s_k
        iv = torch.where(valid, 1.0 / sk2, zero)
        s2 = 1.0 / iv.sum(-1)
        delta = s2 * (d_k * iv).sum(-1)
        den = s2[..., None] + sk2
        pen = torch.log(sk2 / den) + (d_k - delta[..., None]) ** 2 / den
        lnp = torch.where(valid, l_k - 0.5 * pen, zero).sum(-1)
        lnp = torch.where(valid.any(-1), lnp, zero - math.inf).reshape(-1)
        lnp = torch.where(torch.isnan(lnp), zero - math.inf, lnp)
        # the first maximum, in duration then phase order
        top = lnp.max()
        cell = torch.nonzero(lnp == top)[0, 0]
        j = cell % n_phi
        best.append(torch.stack([top, delta.reshape(-1)[cell], torch.sqrt(s2.reshape(-1)[cell]),
                                 t_ref + (j.to(t.dtype) / n_phi) * P,
                                 (cell // n_phi).to(t.dtype)]))
    lnp, delta, sigma, T0, d = torch.stack(best).T
    none = torch.isinf(lnp)
    nan = torch.full_like(lnp, math.nan)
    return dict(Q=torch.where(none, torch.zeros_like(lnp), delta / sigma),
                T0=torch.where(none, nan, T0), depth=torch.where(none, nan, delta),
                sigma=torch.where(none, nan, sigma), lnP=lnp,
                D_idx=torch.where(none, torch.full_like(d, -1.0), d).to(torch.int32))


def _exact_refine(case, seed, lc):
    t, C, z0, Z = _dense(lc)
    P, T0, idx = _candidates(case, seed, lc["t"], lc["inject"])
    Ds = _durations(case)
    M = torch.zeros((len(t), len(P)), dtype=t.dtype, device="cuda")
    ok = 2.0 * Ds[idx] <= P
    for c in np.nonzero(ok)[0]:
        lo = math.floor((lc["t"][0] - T0[c] - Ds[idx[c]]) / P[c]) - 1
        hi = math.ceil((lc["t"][-1] - T0[c] + Ds[idx[c]]) / P[c]) + 1
        for q in range(lo, hi + 1):
            M[:, c] += _template(case["template"], t, T0[c] + float(q) * P[c], Ds[idx[c]])
    W = torch.linalg.solve_triangular(C, M, upper=False)
    depth, var, dlnl = _finish((W * W).sum(0), M.T @ z0, M.T @ Z)
    return dict(depth=depth, var=var, dlnl=dlnl, snr=depth / torch.sqrt(var))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None                       # a dense covariance per curve: minutes
    if kind == "fold":
        if case["n"] * case["n_d"] * case["n_p"] > 7.0e9:
            return None
        return _exact_fold(case, *(_cu(a) for a in _events(case, seed)))
    if case["n"] > 24000 or (kind == "chain" and case["n"] * case["n_d"] * case["n_p"] > 2.0e9):
        return None                       # dense covariance and its inverse
    lc = _curve(case, seed)
    if kind == "refine":
        return _exact_refine(case, seed, lc)
    depth, var, dlnl = _exact_linear(case, lc)
    out = dict(depth=depth, var=var, dlnl=dlnl)
    if kind == "chain":
        # the fold of the exact events in FP64; in mixed precision the library
        # folds events rounded to FP32, whose argmax cell can differ
        out["periodic"] = (_exact_fold(case, _cu(lc["t"]), depth, var, dlnl)
                           if case["precision"] == "fp64" else
                           {a: None for a in ("Q", "T0", "depth", "sigma", "lnP", "D_idx")})
    return out
