"""GPU test of the default phase step: the median spacing selected on the device
is numpy's, for odd and even numbers of spacings, ties, gaps and jitter."""
import numpy as np
import pytest

from paper_2402_06835_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402


def _epochs(n, kind, rng):
    if kind == "two":                      # two distinct spacings, half each
        return np.cumsum(np.where(np.arange(n) % 2 == 0, 1.0, 1.5)) * synth.CADENCE_DAYS
    t = 1000.0 + np.arange(n) * synth.CADENCE_DAYS
    if kind == "gap":
        t[n // 2:] += 1.0
    if kind == "jitter":
        t = np.sort(t + rng.uniform(-0.4, 0.4, n) * synth.CADENCE_DAYS)
    return t


@pytest.mark.parametrize("kind", ["regular", "gap", "jitter", "two"])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 33, 1024, 1025, 1026, 5001, 19440])
def test_default_phase_step_is_the_median_spacing(n, kind):
    rng = np.random.default_rng(n)
    t = _epochs(n, kind, rng)
    step = float(np.median(np.diff(t)))
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    d = rng.normal(0, 1e-3, (1, n))
    args = (cu(t), np.ones(1), cu(d), cu(np.full((1, n), 1e-8)), cu(d * d / 2e-8),
            cu(np.linspace(3.3, 40.2, 7) * step))
    # (the step moves every output: phases, epochs and the gap rule)
    ref = api.nu_periodic_search(*args, phase_step=step)
    got = api.nu_periodic_search(*args)
    for k in ref:
        np.testing.assert_array_equal(got[k].cpu().numpy(), ref[k].cpu().numpy(), err_msg=k)
