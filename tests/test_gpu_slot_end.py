"""The filters of the mixed fold at the end of a regular grid.

A regular grid's epochs may lie up to 1e-3 slot off their slots, the last one
too.  A cell whose last event would fall between the last epoch and its slot
does not have that event, though the cells beside it in a group of phases do.
The curves below put the best cell there: strong events at every period before
the last slot and nothing at the end, and periods within 1e-4 of a whole number
of slots.  The filtered call (many periods) returns, to the bit, what every cell
screened gives: few periods, one duration at a time (items of few cells are not
filtered), and the best duration of each.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_screen import KEYS, _fold  # noqa: E402

EPS = np.array([1e-6, 3e-6, 1e-5, 2e-5, 3e-5, 5e-5, 7e-5, 1e-4])


def _curve(n, m, n_D, last, jitter, seed):
    rng = np.random.default_rng(seed)
    t = np.arange(n, dtype=np.float64)
    t[1:-1] += jitter * rng.uniform(-1, 1, n - 2)
    t[-1] += last
    depth = np.zeros((n_D, n))
    if jitter:
        depth += 0.3 * rng.standard_normal((n_D, n))
    for k in range(1, (n - 1) // m + 1):
        at = n - 1 - k * m
        depth[:, max(at - 4, 0): at + 1] = 10.0
        depth[:, at + 1] = 9.9
    depth *= np.linspace(1.0, 0.9, n_D)[:, None]
    return t, depth, np.ones((n_D, n)), depth ** 2 / 2


def every_cell(t, depth, var, dlnl, periods, dt):
    """The mixed fold with every cell screened (at most 2 304 phases per period):
    the largest ln P over the durations, the first one of equals."""
    assert np.all(periods < 2303 * dt) and len(periods) < 200
    rows = [_fold(api.nu_periodic_search, t, depth[d:d + 1], var[d:d + 1], dlnl[d:d + 1],
                  periods, "mixed", dt) for d in range(len(depth))]
    best = np.argmax([np.where(r["D_idx"] < 0, -np.inf, r["lnP"]) for r in rows], axis=0)
    out = {k: np.choose(best, [r[k] for r in rows]) for k in KEYS}
    out["D_idx"] = np.where(out["D_idx"] < 0, -1, best)
    return out


@pytest.mark.parametrize("jitter", [0.0, 9e-4])
@pytest.mark.parametrize("last", [-9e-4, -5e-4, -1e-4, 0.0, 1e-4, 9e-4])
@pytest.mark.parametrize("n, m, n_D, n_P", [
    (1004, 150, 1, 41000),       # 6.7 epochs per cell (150 cells: not filtered)
    (1004, 150, 6, 41000),       # one warp per period
    (1004, 150, 5, 16),          # the small call's gains
    (1004, 150, 8, 9000), (1004, 150, 20, 4000),
    (1004, 230, 6, 41000),       # 4.4: groups that the gains pass
    (1509, 90, 9, 10000), (2003, 140, 7, 5000), (2003, 60, 12, 8000)])
def test_last_event_beyond_the_last_epoch(n, m, n_D, n_P, last, jitter):
    t, depth, var, dlnl = _curve(n, m, n_D, last, jitter, n + m)
    few = np.concatenate([m - EPS, m + EPS])
    every = every_cell(t, depth, var, dlnl, few, 1.0)
    copies = -(-n_P // len(few))
    got = _fold(api.nu_periodic_search, t, depth, var, dlnl, np.tile(few, copies), "mixed", 1.0)
    for k in KEYS:
        np.testing.assert_array_equal(got[k], np.tile(every[k], copies), err_msg=k)
