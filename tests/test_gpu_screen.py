"""GPU tests of the fold's screens: a screened fold returns what the
evaluation of every cell returns.

The mixed fold of a grid that is not regular runs its exact path (FP64 epochs,
FP32 values) behind the screens of the FP64 fold; the allocation-free entry
point runs the same exact path without them where only the screens' arrays
exceed its fixed scratch.  Both give the same FP32 ln P for a cell, so their
outputs are equal to the bit.
"""
import numpy as np
import pytest

from oracle import periodic
from paper_2402_06835_gb300 import synth
from parity import FP64_TOL, MIXED_SNR_ABS, periodic_compare

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402

KEYS = ("Q", "T0", "depth", "sigma", "lnP", "D_idx")


def cu(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype, device="cuda")


def _grid(n, n_D, seed, kind, gaps=2, consistent=True):
    """Epochs (regular, drifting like barycentric times, or jittered with
    near-coincident pairs), depths that are smooth along the epochs, variances
    with a few outliers, NaN holes, one strong event."""
    rng = np.random.default_rng(seed)
    dt = synth.CADENCE_DAYS
    slots = np.arange(n) + (np.arange(n) * (gaps + 1) // n) * 37
    slots = np.delete(slots, rng.choice(np.arange(2, n - 2), n // 100, replace=False))
    t = slots * dt
    if kind == "drift":
        t = 1500.0 + t + 0.005 * np.sin(2 * np.pi * t / 365.25 + rng.uniform(0, 6))
    elif kind == "jitter":
        t = t + 0.45 * dt * rng.uniform(-1, 1, len(t))
        t[7::101] = t[6::101][: len(t[7::101])] + 0.1 * dt
        t = np.sort(t)
    n = len(t)
    y = rng.standard_normal((n_D, n + 16))
    depth = np.stack([np.convolve(y[d], np.ones(d % 9 + 2) / (d % 9 + 2), "valid")[:n]
                      for d in range(n_D)]) * 2e-4
    var = np.full((n_D, n), 4e-8) * rng.uniform(0.8, 1.2, (n_D, 1))
    var[:, ::211] *= 50.0
    depth[:, n // 3: n // 3 + 9] += 1.5e-3
    dlnl = depth ** 2 / (2 * var) if consistent else rng.uniform(0, 6, (n_D, n))
    depth[:, n // 2: n // 2 + 5] = np.nan
    return t, depth, var, dlnl, dt


def _fold(fn, t, depth, var, dlnl, periods, precision, dt, **kw):
    ft = torch.float64 if precision == "fp64" else torch.float32
    r = fn(cu(t), np.ones(len(depth)), cu(depth, ft), cu(var, ft), cu(dlnl, ft), cu(periods),
           precision=precision, phase_step=dt, **kw)
    return {k: r[k].cpu().numpy() for k in KEYS}


@pytest.mark.parametrize("consistent", [True, False])
@pytest.mark.parametrize("kind", ["drift", "jitter"])
def test_mixed_irregular_screen_equals_every_cell(kind, consistent):
    t, depth, var, dlnl, dt = _grid(50000, 12, 3, kind, consistent=consistent)
    span = t[-1] - t[0]
    periods = np.concatenate([span / np.array([700.3, 120.7, 33.1, 31.9, 17.2, 9.1, 6.4]),
                              np.linspace(span / 5, span / 2, 17), [40 * dt, 100.5 * dt]])
    # the unscreened path: only the screens' arrays exceed the fixed scratch
    every = _fold(api.nu_periodic_search_noalloc, t, depth, var, dlnl, periods, "mixed", dt)
    got = _fold(api.nu_periodic_search, t, depth, var, dlnl, periods, "mixed", dt)
    for k in KEYS:
        np.testing.assert_array_equal(got[k], every[k], err_msg=k)


@pytest.mark.parametrize("kind, precision, n, n_D", [
    ("regular", "fp64", 15500, 14), ("drift", "fp64", 15500, 14), ("jitter", "fp64", 15500, 14),
    ("regular", "mixed", 33000, 13), ("drift", "mixed", 33000, 13),
    ("regular", "fp64", 70000, 3), ("regular", "mixed", 130000, 3),
    ("regular", "fp64", 190000, 1), ("drift", "mixed", 350000, 1)])
def test_filters_equal_every_cell_screened(kind, precision, n, n_D):
    """The filters over groups of cells drop nothing that could win: on grids
    whose filter tables (and only those) exceed the fixed scratch, the
    allocation-free entry point screens every cell.  Periods from 1.3 to 600
    epochs per cell, each filter's range and its limits."""
    t, depth, var, dlnl, dt = _grid(n, n_D, 5 + n_D, kind)
    span = t[-1] - t[0]
    rng = np.random.default_rng(1)
    K = np.concatenate([np.exp(rng.uniform(np.log(1.3), np.log(30.0), 90)),
                        [5.4, 5.6, 21.9, 22.1, 50.0, 150.0, 600.0]])
    periods = np.concatenate([span / K, [200 * dt, 1000.5 * dt]])
    every = _fold(api.nu_periodic_search_noalloc, t, depth, var, dlnl, periods, precision, dt)
    got = _fold(api.nu_periodic_search, t, depth, var, dlnl, periods, precision, dt)
    for k in KEYS:
        np.testing.assert_array_equal(got[k], every[k], err_msg=k)
    # and with two warps or one per period instead of a block
    for copies in (70, 410):
        got = _fold(api.nu_periodic_search, t, depth, var, dlnl, np.tile(periods, copies),
                    precision, dt)
        for k in KEYS:
            np.testing.assert_array_equal(got[k], np.tile(every[k], copies), err_msg=k)


@pytest.mark.parametrize("kind, precision", [("regular", "fp64"), ("drift", "fp64"),
                                             ("jitter", "fp64"), ("drift", "mixed"),
                                             ("jitter", "mixed")])
@pytest.mark.parametrize("n_D", [1, 3, 11])
def test_screened_fold_against_oracle(kind, n_D, precision):
    """The paths whose exact events take their epochs in FP64 (the mixed fold of
    a regular grid takes them from its fixed-point walk instead)."""
    t, depth, var, dlnl, dt = _grid(1500, n_D, 17 + n_D, kind)
    if precision == "mixed":
        depth, var, dlnl = (a.astype(np.float32).astype(np.float64) for a in (depth, var, dlnl))
    span = t[-1] - t[0]
    periods = np.concatenate([span / np.array([60.2, 40.1, 25.3, 14.9, 11.1]),
                              np.linspace(span / 9, 0.8 * span, 60), np.arange(40, 44) * dt])
    ora = periodic.periodic_search(t, depth, var, dlnl, periods, dt)
    got = _fold(api.nu_periodic_search, t, depth, var, dlnl, periods, precision, dt)
    tol, qt = (FP64_TOL, FP64_TOL) if precision == "fp64" else (1e-4, MIXED_SNR_ABS)
    periodic_compare(got, ora, t, depth, var, dlnl, periods, dt, tol, qt,
                     periodic.fold_period, max_reeval=len(periods),
                     q_abs=precision == "mixed")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_of_regular_and_irregular_curves_equals_single_calls(precision):
    """One batch of both kinds of grid: every curve as by the single calls."""
    dt = synth.CADENCE_DAYS
    Ds = np.array([0.02, 0.045, 0.07, 0.09, 0.11])
    periods = np.linspace(0.11, 0.9, 90)
    curves = []
    for c, (n, drift) in enumerate([(400, 0.0), (517, 0.02), (450, 0.0), (611, 0.03)]):
        lc = synth.small_curve(n=n, seed=50 + c, gap=30, inject=(2.5e-3, 1.0 / 24.0, 0.37))
        t = lc.t + drift * dt * np.sin(np.arange(n) / 3.0)
        curves.append((t, lc.y, lc.diag_var, lc.terms))
    res = api.nu_batch_search(curves, Ds, periods, k=2, precision=precision, phase_step=dt)
    assert res["status"] == [0] * len(curves)
    for c, (t, y, dv, terms) in enumerate(curves):
        X = np.stack([np.ones_like(t), t], axis=1)
        f = api.nu_gp_factor(cu(t), cu(dv), terms, cu(X), cu(y))
        d, v, l = api.nu_linear_search(f, cu(t), Ds, precision=precision)
        one = api.nu_periodic_search(cu(t), Ds, d, v, l, cu(periods), precision=precision,
                                     phase_step=dt)
        assert np.array_equal(res["D_idx"][c].cpu().numpy(), one["D_idx"].cpu().numpy())
        for k in ("Q", "T0", "lnP", "depth", "sigma"):
            a, b = res[k][c].cpu().numpy(), one[k].cpu().numpy()
            np.testing.assert_allclose(a, b, rtol=1e-9 if precision == "fp64" else 1e-5,
                                       atol=0, err_msg=f"{k} of curve {c}")
