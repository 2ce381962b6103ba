"""The table form of the Legendre stage at the edges of its kernels, against a
plan of the native FP64 kernels (the double-float recurrence is no reference: its
own error reaches 1.7e-12 of the largest value near the poles): row counts next to the pairs, groups of four and chunks of 96
rows (lmax + 1 = 2 rows), ring pairs that fill part of a tile of 32, band limits
that end inside a pair, a group or a chunk, and two maps in one launch with one
of them stopped early. Bar 1e-12 of the largest output: 48-bit products summed
over at most 512 terms err by 1e-13, a dropped row or tile by far more."""
import numpy as np
import pytest

from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


def plan(nside, lmax, **kw):
    npix = 12 * nside * nside
    cl = 1.0 / (1.0 + np.arange(lmax + 1)) ** 2
    nv = 1.0 + 0.5 * np.cos(np.arange(npix))
    return wf.Plan(nside, lmax, cl, nv, opts=wf.options(**kw))


@pytest.mark.parametrize("nside,lmax,lsht", [(1, 0, 0), (1, 3, 2), (8, 31, 31), (16, 6, 5), (16, 63, 40), (64, 189, 189),
                                             (64, 190, 190), (64, 191, 188), (64, 192, 191), (128, 385, 193),
                                             (256, 255, 255), (512, 70, 70), (1024, 40, 37)])
def test_table_against_native(nside, lmax, lsht):
    import torch
    npix, nalm = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    rng = np.random.default_rng(nside + lmax)
    a = rng.standard_normal(nalm) + 1j * rng.standard_normal(nalm)
    a[:lmax + 1].imag = 0.0
    f = rng.standard_normal(npix)
    got = []
    for prec in (wf.WF_PREC_FP64, wf.WF_PREC_FP64_NATIVE):
        P = plan(nside, lmax, precision=prec)
        assert (P.legendre_table(lmax)[0] > 0) == (prec == wf.WF_PREC_FP64)
        ad, fd = torch.from_numpy(a).cuda(), torch.from_numpy(f).cuda()
        m = torch.zeros(npix, dtype=torch.float64, device="cuda")
        t = torch.zeros(nalm, dtype=torch.complex128, device="cuda")
        s = torch.zeros(nalm, dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        P.alm2map(lsht, ad.data_ptr(), m.data_ptr())
        P.map2alm(lsht, fd.data_ptr(), t.data_ptr())
        recs = P.iterate(fd.data_ptr(), s.data_ptr(), 2.5, lsht, 3)
        torch.cuda.synchronize()
        got.append([x.cpu().numpy() for x in (m, t, s)] +
                   [np.array([[r["chi2_prior"], r["chi2_noise"], r["incr2"], r["norm2"]] for r in recs])])
        P.close()
    for x, y in zip(*got):
        assert np.max(np.abs(x - y)) <= 1e-12 * max(np.max(np.abs(y)), 1e-300)


def test_pair_with_one_map_stopped_early():
    """Two right-hand sides of very different scale share the launches; each result is its single solve's, bit for bit."""
    nside, lmax = 32, 95
    rng = np.random.default_rng(3)
    d = rng.standard_normal((3, 12 * nside * nside)) * np.array([[1.0], [30.0], [0.01]])
    P = plan(nside, lmax, tol=1e-5, max_iter=400)
    out, st, _ = P.solve_batch(d)
    for i in range(3):
        alone, s1, _, _ = P.solve(d[i])
        assert s1["iters"] == st[i]["iters"]
        assert np.array_equal(alone, out[i])
    P.close()
