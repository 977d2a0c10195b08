"""Scratch of the batch search: the lists of its (curve, period) items are bounded
(2^22 items, 1 GB), a large batch goes through them in passes over its curves or
over a curve's periods and returns what a small one returns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api, synth  # noqa: E402
from test_gpu_fold_passes import _PoolHigh  # noqa: E402
from test_gpu_screen import KEYS  # noqa: E402


def _curves(n_lc):
    dt = synth.CADENCE_DAYS
    out = []
    for c in range(n_lc):
        lc = synth.small_curve(n=140 + 3 * c, seed=70 + c, gap=10, inject=(2.5e-3, 1.0 / 24.0, 0.07))
        drift = 0.03 if c % 3 == 1 else 0.0
        out.append((lc.t + drift * dt * np.sin(np.arange(len(lc.t)) / 3.0), lc.y, lc.diag_var,
                    lc.terms))
    return out, dt


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n_lc, n_P", [(24, 400_001), (2, 4_900_000)])
def test_large_batch_in_bounded_scratch(precision, n_lc, n_P):
    curves, dt = _curves(n_lc)
    Ds = np.array([0.03])
    periods = np.linspace(0.03, 0.11, n_P)
    high = _PoolHigh()
    torch.cuda.synchronize()
    high.reset()
    big = api.nu_batch_search(curves, Ds, periods, k=2, precision=precision, phase_step=dt)
    # 230 bytes x 2^22 and 88 per period; for all items at once 2.2 GB and more
    assert high.read() < 1.6e9
    some = np.r_[0:n_P:20011, n_P - 1]
    few = api.nu_batch_search(curves, Ds, periods[some], k=2, precision=precision, phase_step=dt)
    assert big["status"] == few["status"] == [0] * n_lc
    at = torch.as_tensor(some, device="cuda")
    for k in KEYS:
        np.testing.assert_array_equal(big[k][:, at].cpu().numpy(), few[k].cpu().numpy(),
                                      err_msg=k)
