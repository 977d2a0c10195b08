"""Items of few cells per lane screen every cell, the others filter: periods on
both sides of the line, and cells of up to 300 epochs, give what calls small
enough to screen every cell give, to the bit, with eight, two and one warp per
period (nine, nine and twenty cells per lane)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_screen import KEYS, _fold, _grid  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["regular", "drift"])
@pytest.mark.parametrize("n_D", [1, 3])
def test_periods_about_the_line(kind, precision, n_D):
    t, depth, var, dlnl, dt = _grid(9000, n_D, 61 + n_D, kind)
    span = t[-1] - t[0]
    lines = np.concatenate([[288 * nw // n_D + d for d in (-1, 0, 0.5, 1, 2)] for nw in (8, 2)]
                           + [[640 // n_D + d for d in (-1, 0, 0.5, 1, 2)]])
    base = np.concatenate([lines * dt, 30.3 * dt * np.arange(1, 9), span / np.arange(2.2, 9)])
    few = _fold(api.nu_periodic_search, t, depth, var, dlnl, base, precision, dt)
    assert len(base) * 9100 * n_D < 2.4e7
    for n_P in (4000 // n_D, 5900, 41000):
        copies = -(-n_P // len(base))
        got = _fold(api.nu_periodic_search, t, depth, var, dlnl, np.tile(base, copies),
                    precision, dt)
        for k in KEYS:
            np.testing.assert_array_equal(got[k], np.tile(few[k], copies), err_msg=k)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["regular", "drift"])
@pytest.mark.parametrize("n_P, long", [(4990, 1.0), (5800, 1.0), (5800, 0.3), (41000, 0.05),
                                       (41000, 1.0)])
def test_many_long_items(kind, precision, n_P, long):
    """Items of 22 or more epochs per cell take blocks beside the warps of the
    others up to 5 000 of them (a tenth of the items, beside one warp each), and
    warps beyond."""
    t, depth, var, dlnl, dt = _grid(6500, 20, 71, kind)
    span = t[-1] - t[0]
    n = 60
    n_long = int(round(long * n))
    base = np.concatenate([span / np.linspace(24, 90, n_long),
                           span / np.linspace(3, 18, n - n_long)])
    few = [_fold(api.nu_periodic_search, t, depth, var, dlnl, base[lo:lo + 30], precision, dt)
           for lo in (0, 30)]
    copies = -(-n_P // n)
    got = _fold(api.nu_periodic_search, t, depth, var, dlnl, np.tile(base, copies), precision, dt)
    for k in KEYS:
        want = np.concatenate([f[k] for f in few])
        np.testing.assert_array_equal(got[k], np.tile(want, copies), err_msg=k)
