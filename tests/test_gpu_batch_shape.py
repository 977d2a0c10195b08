"""The batch fold's tuned launch shape does not carry over to another kind of
batch: after a small batch of short curves, whose cells are all short, the long
cells of a batch of long curves still take blocks of eight warps."""
import json

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api, synth  # noqa: E402


def _kernels(path, call):
    for _ in range(2):                 # (the first session of a process may see none)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU,
                                                torch.profiler.ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        prof.export_chrome_trace(str(path))
        with open(path) as f:
            events = json.load(f)["traceEvents"]
        names = {e["name"] for e in events if e.get("cat") == "kernel"}
        if names:
            break
    return names


@pytest.mark.parametrize("precision, block", [("fp64", "k_fold_cells<double, 8"),
                                              ("mixed", "k_fold_slot_cells<8")])
@pytest.mark.parametrize("n_D", [1, 4, 9])
def test_long_cells_take_blocks_after_a_batch_of_short_ones(precision, block, n_D, tmp_path):
    dt = synth.CADENCE_DAYS
    Ds = np.linspace(0.02, 0.06, n_D)

    def batch(n, n_lc, lo, hi, n_P):
        curves = [(lc.t, lc.y, lc.diag_var, lc.terms)
                  for lc in (synth.small_curve(n=n, seed=90 + c, gap=10) for c in range(n_lc))]
        api.nu_batch_search(curves, Ds, np.linspace(lo, hi, n_P), k=1, precision=precision,
                            phase_step=dt)
    batch(300, 64, 0.15, 0.3, 1000)                        # 1.4 to 2.8 epochs per cell
    long = lambda: batch(6000, 4, 0.12, 0.3, 2000)         # 28 to 70
    long()                                                 # (tunes, if it has to)
    names = _kernels(tmp_path / "trace", long)
    if not names:
        pytest.skip("the profiler reports no kernels here")
    assert any(block in n for n in names), sorted(n for n in names if "k_fold" in n)
