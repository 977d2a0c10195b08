"""Scratch of the periodic search: bounded however many periods a call has (the
periods go through their table and lists in passes), and the allocation-free
call's fixed scratch holds filter tables wherever the records leave room.
Passes and reduced tables return what one pass with all tables returns."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_screen import KEYS, _fold, _grid  # noqa: E402


def _launched(call):
    n0 = api.launch_count()
    r = call()
    return r, api.launch_count() - n0


@pytest.mark.parametrize("kind, precision, n, n_D, n_P", [
    ("regular", "fp64", 19440, 10, 20000),     # all tables, several passes
    ("drift", "fp64", 19440, 10, 9001),
    ("regular", "mixed", 19440, 16, 20000), ("drift", "mixed", 19440, 16, 20000),
    ("regular", "fp64", 19440, 12, 3000),      # the gains' tables only
    ("jitter", "fp64", 19440, 12, 3000),
    ("drift", "mixed", 24000, 17, 2500),
    ("regular", "fp64", 2000, 4, 100001), ("regular", "mixed", 2000, 4, 100001)])
def test_noalloc_keeps_the_filters(kind, precision, n, n_D, n_P):
    t, depth, var, dlnl, dt = _grid(n, n_D, 41 + n_D, kind)
    span = t[-1] - t[0]
    periods = np.linspace(span / 60, 0.6 * span, n_P)
    args = (t, depth, var, dlnl, periods, precision, dt)
    few = (t, depth, var, dlnl, periods[:40], precision, dt)
    want = _fold(api.nu_periodic_search, *args)
    got, launched = _launched(lambda: _fold(api.nu_periodic_search_noalloc, *args))
    for k in KEYS:
        np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    _, unfiltered = _launched(lambda: _fold(api.nu_periodic_search_noalloc, *few))
    assert launched >= unfiltered + 2          # at least the two tables of the gains


class _PoolHigh:
    """High-water mark of the device's default memory pool (the library's; the
    tensors' allocator does not use it)."""
    USED_HIGH = 8

    def __init__(self):
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def reset(self):
        zero = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, self.USED_HIGH,
                                               ctypes.byref(zero)) == 0

    def read(self):
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, self.USED_HIGH, ctypes.byref(v)) == 0
        return v.value


@pytest.mark.parametrize("kind, precision", [("regular", "fp64"), ("regular", "mixed"),
                                             ("drift", "mixed")])
def test_scratch_does_not_grow_with_the_periods(kind, precision):
    """3 million periods: less than 300 MB (2^19 periods of 290 bytes and a list's
    counters; a table and lists for all of them take 1.3 GB)."""
    t, depth, var, dlnl, dt = _grid(260, 1, 3, kind)
    span = t[-1] - t[0]
    periods = np.linspace(0.2 * span, 0.7 * span, 3_000_000)
    high = _PoolHigh()
    torch.cuda.synchronize()
    high.reset()
    got = _fold(api.nu_periodic_search, t, depth, var, dlnl, periods, precision, dt)
    assert high.read() < 300e6
    some = np.r_[0:3_000_000:9973, 524287:524290]
    part = _fold(api.nu_periodic_search, t, depth, var, dlnl, periods[some], precision, dt)
    for k in KEYS:
        np.testing.assert_array_equal(got[k][some], part[k], err_msg=k)
