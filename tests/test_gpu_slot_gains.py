"""Small calls of the mixed fold on a regular grid bound their cells by the gains
alone: they and the calls with all tables return, to the bit, what every cell
screened gives, over few and many epochs per cell, one to nine durations, holes,
gains that no bound covers (1e25) and gains below zero."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_screen import KEYS, _fold, _grid  # noqa: E402
from test_gpu_slot_end import every_cell  # noqa: E402


@pytest.mark.parametrize("gains", ["consistent", "free", "odd", "negative"])
@pytest.mark.parametrize("n, n_D", [(1301, 1), (1800, 2), (2600, 5), (3500, 9), (20000, 4)])
def test_small_call_equals_every_cell(n, n_D, gains):
    t, depth, var, dlnl, dt = _grid(n, n_D, 81 + n_D, "regular", consistent=gains == "consistent")
    if gains == "odd":
        dlnl[:, ::401] = 1e25
        var[:, 5::307] *= 1e4
    if gains == "negative":
        dlnl = dlnl - 4.0
    span = t[-1] - t[0]
    top = min(0.8 * span, 2300 * dt)
    periods = np.concatenate([np.linspace(span / 60, top, 60), [200 * dt, 100.5 * dt, top]])
    every = every_cell(t, depth, var, dlnl, periods, dt)
    small = _fold(api.nu_periodic_search, t, depth, var, dlnl, periods, "mixed", dt)
    copies = int(1.3e8 / (span / dt * n_D * len(periods))) + 1
    large = _fold(api.nu_periodic_search, t, depth, var, dlnl, np.tile(periods, copies), "mixed", dt)
    for k in KEYS:
        np.testing.assert_array_equal(small[k], every[k], err_msg=k)
        np.testing.assert_array_equal(large[k], np.tile(every[k], copies), err_msg=k)
