"""The batched engine's ring stage at the ends of its range: grids whose rings
are all shorter than the block (one FFT class, short twiddle tables), slot
counts that leave a group part full, and Nside 2048, whose longest rings run one
to a CTA where the others run in pairs. Fixed iterations of a few maps against
the FP64 plan of the same problem. Bar 1e-6 relative L2, the mixed engine's."""
import numpy as np
import pytest

from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,nrhs", [(1, 3, 1), (2, 7, 3), (4, 15, 9), (64, 130, 5), (2048, 40, 2)])
def test_few_iterations_against_fp64(nside, lmax, nrhs):
    npix = 12 * nside * nside
    rng = np.random.default_rng(nside)
    cl = np.where(np.arange(lmax + 1) >= 2, 1.0 / (1.0 + np.arange(lmax + 1)) ** 2, 0.0)
    nv = 0.5 + rng.random(npix)
    mask = (rng.random(npix) > 0.1).astype(np.uint8)
    d = rng.standard_normal((nrhs, npix))
    out = []
    for prec in (wf.WF_PREC_MIXED, wf.WF_PREC_FP64):
        P = wf.Plan(nside, lmax, cl, nv, mask, wf.options(precision=prec, tol=0.0, max_iter=4, cooling=0,
                                                          batch_slots=nrhs))
        alm, st, _ = P.solve_batch(d)
        assert [s["iters"] for s in st] == [4] * nrhs
        out.append(alm)
        P.close()
    for i in range(nrhs):
        assert np.linalg.norm(out[0][i] - out[1][i]) <= 1e-6 * np.linalg.norm(out[1][i])
