"""nu_periodic_refine gives a candidate one, two or eight warps by the number
of candidates: both sides of each boundary, on curves shorter than one segment
per thread and longer, against the oracle's dense fit."""
import numpy as np
import pytest

from oracle import linear
from paper_2402_06835_gb300 import synth
from parity import FP64_TOL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2402_06835_gb300 import api  # noqa: E402
from test_gpu_refine import candidate_set, cu, errors, gpu_refine, oracle_refine  # noqa: E402


@pytest.mark.parametrize("n", [150, 2200])
@pytest.mark.parametrize("kind", ["box", "limb_quad"])
def test_candidates_around_the_warp_boundaries(n, kind):
    lc = synth.small_curve(n=n, seed=5, p_rot=1.3, sigma=4e-3, sigma_w=1e-3,
                           inject=(3e-3, 1.0 / 24.0, 0.41))
    Ds = np.array([0.03, 1.0 / 24.0, 0.055])
    model = linear.DenseModel(lc.t, lc.y, lc.diag_var, lc.terms, lc.X)
    cands = candidate_set(lc.t, len(Ds), np.random.default_rng(8), n_random=292)
    o = oracle_refine(model, cands, Ds, kind, 0.3)
    f = api.nu_gp_factor(cu(lc.t), cu(lc.diag_var), lc.terms, cu(lc.X), cu(lc.y))
    for c in (1, 76, 77, 304, 305):
        lo = len(cands) - c                     # the special ones are last
        err = errors(gpu_refine(f, cands[lo:], Ds, kind, 0.3),
                     {k: np.asarray(v)[lo:] for k, v in o.items()})
        assert max(err["depth"], err["var"], err["dlnl"], err["snr"]) <= FP64_TOL, (c, err)
