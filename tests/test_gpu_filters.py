"""The filters drop nothing that could win: calls large enough for their tables
return what calls small enough to screen every cell (or, on regular grids in
mixed precision, to bound them by their gains alone) return, to the bit.  The number of
kernels launched shows that the filter tables are built in the one and not in
the other (three launches), so that neither side silently takes the other's path.
Periods from 1.3 to 600 epochs per cell, each filter's range and its limits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_screen import KEYS, _fold, _grid  # noqa: E402


def _counted(*args):
    n0 = api.launch_count()
    r = _fold(api.nu_periodic_search, *args)
    return r, api.launch_count() - n0


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["regular", "drift", "jitter"])
@pytest.mark.parametrize("n, n_D, n_P, scale", [
    (15500, 14, 330, 1.0), (15500, 6, 700, 1.0), (9000, 2, 1450, 1.0), (70000, 1, 1000, 1.0),
    (6000, 5, 1500, 300.0)])          # (the last: gains beyond the FP16 range)
def test_block_filters_equal_every_cell_screened(kind, precision, n, n_D, n_P, scale):
    """Eight warps per period, with the filters and without."""
    t, depth, var, dlnl, dt = _grid(n, n_D, 29 + n_D, kind)
    depth, dlnl = depth * scale, dlnl * scale * scale
    span = t[-1] - t[0]
    steps = span / dt * n_D
    if kind == "regular" and precision == "mixed":       # the slot path
        line = 6e7 if steps < 4e4 else 2.4e7
        n_P = max(n_P, int(1.1 * line / steps))          # (two warps in two of the cases)
    else:
        line = 4e7 if n_D == 1 else 2.4e7
    rng = np.random.default_rng(2)
    K = np.exp(rng.uniform(np.log(1.3), np.log(40.0), n_P))
    K[:12] = [5.4, 5.6, 3.7, 3.9, 16.4, 18.6, 21.9, 22.1, 50.0, 150.0, 600.0, 31.9]
    periods = span / rng.permutation(K)
    periods[5:7] = 200 * dt, 1000.5 * dt
    whole, launched = _counted(t, depth, var, dlnl, periods, precision, dt)
    few = int(line / steps * 0.9)
    assert 0 < few < n_P
    for lo in range(0, n_P, few):
        part, launched_part = _counted(t, depth, var, dlnl, periods[lo:lo + few], precision, dt)
        assert launched >= launched_part + 3
        for key in KEYS:
            np.testing.assert_array_equal(whole[key][lo:lo + few], part[key], err_msg=key)
