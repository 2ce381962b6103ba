"""The batched engine's ring stage at Nside 1024, whose longest Bluestein rings run one to a CTA and the others in
pairs, with slots that fill and that part fill a group. Fixed iterations against the FP64 plan of the same problem.
Bar 1e-6 relative L2, the mixed engine's."""
import numpy as np
import pytest

from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax,nrhs", [(30, 4), (47, 5)])
def test_few_iterations_at_nside_1024(lmax, nrhs):
    nside = 1024
    npix = 12 * nside * nside
    rng = np.random.default_rng(lmax)
    cl = np.where(np.arange(lmax + 1) >= 2, 1.0 / (1.0 + np.arange(lmax + 1)) ** 2, 0.0)
    nv = 0.5 + rng.random(npix)
    mask = (rng.random(npix) > 0.1).astype(np.uint8)
    d = rng.standard_normal((nrhs, npix))
    out = []
    for prec in (wf.WF_PREC_MIXED, wf.WF_PREC_FP64):
        P = wf.Plan(nside, lmax, cl, nv, mask, wf.options(precision=prec, tol=0.0, max_iter=4, cooling=0,
                                                          batch_slots=nrhs))
        alm, _, _ = P.solve_batch(d)
        out.append(alm)
        P.close()
    for i in range(nrhs):
        assert np.linalg.norm(out[0][i] - out[1][i]) <= 1e-6 * np.linalg.norm(out[1][i])
