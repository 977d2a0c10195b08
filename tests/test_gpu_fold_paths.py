"""The fold of many periods (filters, survivors packed into warps, two warps per
period) returns what the same periods give in calls small enough to screen
every cell and evaluate survivors in place (eight warps per period): to the
bit, over few and many epochs per cell."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_screen import KEYS, _fold, _grid  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["regular", "drift", "jitter"])
@pytest.mark.parametrize("n, n_D, n_P", [(3001, 1, 14000), (2600, 3, 4000), (1203, 12, 2500)])
def test_large_call_equals_small_calls(kind, precision, n, n_D, n_P):
    t, depth, var, dlnl, dt = _grid(n, n_D, 11 + n_D, kind)
    span = t[-1] - t[0]
    periods = np.concatenate([np.linspace(span / 70, span / 15, n_P // 4),
                              np.linspace(0.9 * span, span / 15, n_P - n_P // 4)])
    whole = _fold(api.nu_periodic_search, t, depth, var, dlnl, periods, precision, dt)
    for lo in range(0, n_P, n_P // 10):
        part = _fold(api.nu_periodic_search, t, depth, var, dlnl,
                     periods[lo:lo + 150], precision, dt)
        for key in KEYS:
            a = whole[key][lo:lo + 150]
            assert np.array_equal(a, part[key], equal_nan=True), (lo, key)
