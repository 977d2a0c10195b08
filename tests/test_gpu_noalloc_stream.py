"""The allocation-free fold runs on the caller's stream alone and creates no
stream of its own: its callers may not allocate while they run.  The calls here
hold a list of long cells, which nu_periodic_search folds on a side stream."""
import json

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_screen import KEYS, _fold, _grid  # noqa: E402


def _streams(path, call):
    """Streams of the fold's kernels during call() (empty if the profiler saw none;
    its first session in a process may)."""
    for _ in range(2):
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU,
                                                torch.profiler.ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        prof.export_chrome_trace(str(path))
        with open(path) as f:
            events = json.load(f)["traceEvents"]
        found = {e["args"]["stream"] for e in events
                 if e.get("cat") == "kernel" and "nu::" in e.get("name", "")}
        if found:
            break
    return found


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_noalloc_uses_one_stream(precision, tmp_path):
    t, depth, var, dlnl, dt = _grid(1203, 12, 23, "regular")
    span = t[-1] - t[0]
    periods = np.concatenate([np.linspace(span / 70, span / 15, 1500),
                              np.linspace(0.9 * span, span / 15, 4500)])
    out = {}

    def run(fn):
        out[fn] = _fold(fn, t, depth, var, dlnl, periods, precision, dt)
    forked = _streams(tmp_path / "a", lambda: run(api.nu_periodic_search))
    if not forked:
        pytest.skip("the profiler reports no kernels here")
    assert len(forked) == 2                   # (these calls do have a list)
    assert len(_streams(tmp_path / "b", lambda: run(api.nu_periodic_search_noalloc))) == 1
    for k in KEYS:
        np.testing.assert_array_equal(out[api.nu_periodic_search][k],
                                      out[api.nu_periodic_search_noalloc][k], err_msg=k)
