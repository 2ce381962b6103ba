"""Spectra that reach the ends of the range of a double."""
import numpy as np
import pytest

from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [wf.WF_PREC_FP64, wf.WF_PREC_FP64_NATIVE])
def test_joint_filter_of_a_spectrum_that_fades_through_the_subnormals(precision):
    """C_l falls through the subnormal numbers to 0, as a Gaussian cut-off does. Modes of such a C_l come out as 0, or
    next to it; the others as with C_l = 0 there (their own arithmetic is the same: bar 1e-12 relative L2)."""
    nside, lmax = 8, 20
    npix = 12 * nside * nside
    rng = np.random.default_rng(4)
    l = np.arange(lmax + 1)
    faint = {14: 1e-300, 15: 2.5e-308, 16: 7e-309, 17: 5e-309, 18: 1e-310, 19: 5e-324, 20: 0.0}
    cl = np.where(l >= 2, 1.0 / (1.0 + l) ** 2, 0.0)
    cut = cl.copy()
    for k, v in faint.items():
        cl[k], cut[k] = v, 0.0
    nv = [0.5 + rng.random(npix) for _ in range(2)]
    d = rng.standard_normal((2, npix))
    got = []
    for c in (cl, cut):
        M = wf.Multi(nside, lmax, c, nv, opts=wf.options(precision=precision, tol=0.0, max_iter=8, cooling=0))
        alm, st, status, rec = M.solve(d, history=8)
        assert st["iters"] == 8 and np.all(np.isfinite([r["chi2_prior"] for r in rec]))
        got.append((alm.copy(), [r["chi2"] for r in rec]))
        M.close()
    ls = np.concatenate([np.arange(m, lmax + 1) for m in range(lmax + 1)])
    assert np.max(np.abs(got[0][0][ls >= 14])) < 1e-290
    assert np.linalg.norm(got[0][0] - got[1][0]) <= 1e-12 * np.linalg.norm(got[1][0])
    # chi^2 of 14 faint modes with s = C_l x: C_l x^2, nothing
    np.testing.assert_allclose(got[0][1], got[1][1], rtol=1e-12)


def test_polarised_filter_far_below_unit_scale():
    """Spectra and noise times 2^-514, data times 2^-257: the same filter scaled by 2^-257, although the determinants of
    Eq. 4 (about 2^-1028) are subnormal. Bar 1e-11: their last bit is 2^-46 of them (1.4e-14), met a few times in each of
    five iterations."""
    nside, lmax = 4, 9
    npix = 12 * nside * nside
    rng = np.random.default_rng(6)
    tt = 1.0 / (1.0 + 0.1 * np.arange(lmax + 1))
    cls = np.stack([tt, 0.8 * tt, 0.7 * tt, 0.3 * tt])
    cov = np.tile([1.0, 1.2, 0.1, 1.1], (npix, 1)) * (1.0 + rng.random((npix, 1)))
    d = rng.standard_normal((3, npix))
    out = []
    for e in (0, -257):
        P = wf.Pol(nside, lmax, list(cls * 2.0 ** (2 * e)), cov * 2.0 ** (2 * e),
                   opts=wf.options(precision=wf.WF_PREC_FP64_NATIVE, tol=0.0, max_iter=5, cooling=0))
        alm, st, _, _ = P.solve(d * 2.0 ** e)
        assert st["iters"] == 5
        out.append(alm * 2.0 ** -e)
        P.close()
    assert np.linalg.norm(out[1] - out[0]) <= 1e-11 * np.linalg.norm(out[0])
