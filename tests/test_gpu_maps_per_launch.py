"""Several maps per ring-stage and Legendre launch: more maps than a launch takes
(four and two), on the double-float forms, against the oracle's joint iteration
over a fixed count. Bar 1e-10 relative L2, the FP64 paths' parity bar."""
import numpy as np
import pytest

from oracle import multi as MU
from oracle import oracle as O
from paper_1211_0585_gb300 import wf

from gpu_util import FP64_PATHS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", list(FP64_PATHS))
@pytest.mark.parametrize("ndet", [4, 5, 9])
def test_many_detectors_match_oracle(ndet, prec):
    nside, lmax = 4, 11
    rng = np.random.default_rng(ndet)
    npix = 12 * nside * nside
    ell = np.arange(lmax + 1)
    cl = np.where(ell >= 2, 1.0 / (1.0 + ell) ** 2, 0.0)
    beams = [np.exp(-0.5 * ell * (ell + 1) * (0.02 * k) ** 2) for k in range(ndet)]
    var = [0.05 * (1 + k) * (1 + rng.random(npix)) for k in range(ndet)]
    masks = [(rng.random(npix) > 0.2).astype(np.uint8) for _ in range(ndet)]
    ds = [rng.standard_normal(npix) for _ in range(ndet)]
    opts = dict(tol=0.0, max_iter=25, l_iter0=4)
    ores = MU.solve_multi(nside, lmax, cl, beams, var, masks, ds, O.Options(**opts, band_limit=False))
    M = wf.Multi(nside, lmax, cl, var, masks, beams, wf.options(**FP64_PATHS[prec], **opts))
    alm, st, _, recs = M.solve(ds, history=26)
    assert st["iters"] == ores.iters == 25
    assert O.rel_l2(alm, ores.alm, lmax) < 1e-10
    for r, h in zip(recs, ores.history):
        assert r["chi2"] == pytest.approx(h["chi2"], rel=1e-10)
    M.close()
