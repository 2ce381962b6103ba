"""The polarised transform pair in double-float against the native FP64 form of
the same plan (its own spin-2 and ring kernels), at sizes that meet the edges
of the double-float kernels: fewer ring pairs than a warp, a CTA or a chunk of
them, lmax next to the analysis' chunks of 16 and 64 values of l, odd row
counts, and m < 2 (rows without an l >= 2). Bar: 1e-11 of the largest output,
four digits above the forms' own errors (1e-13 at these sizes) and far below
single precision, which a lost low part would leave."""
import numpy as np
import pytest

from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax", [(1, 1), (1, 4), (2, 2), (4, 15), (4, 16), (8, 17), (16, 63), (32, 127),
                                        (64, 255), (64, 256), (128, 257), (128, 321)])
def test_pol_pair_against_native(nside, lmax):
    import torch
    npix, nalm = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    rng = np.random.default_rng(nside * 10000 + lmax)
    a = rng.standard_normal((3, nalm)) + 1j * rng.standard_normal((3, nalm))
    a[:, :lmax + 1].imag = 0.0
    f = rng.standard_normal((3, npix))
    got = []
    for prec in (wf.WF_PREC_FP64, wf.WF_PREC_FP64_NATIVE):
        P = wf.Pol(nside, lmax, [np.ones(lmax + 1)] * 3 + [np.zeros(lmax + 1)], np.tile([1.0, 1.0, 0.0, 1.0], (npix, 1)),
                   opts=wf.options(precision=prec))
        ad, fd = torch.from_numpy(a).cuda(), torch.from_numpy(f).cuda()
        md = torch.zeros(3, npix, dtype=torch.float64, device="cuda")
        td = torch.zeros(3, nalm, dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        P.alm2map(ad.data_ptr(), md.data_ptr())
        P.map2alm(fd.data_ptr(), td.data_ptr())
        torch.cuda.synchronize()
        got.append((md.cpu().numpy(), td.cpu().numpy()))
        P.close()
    for x, y in zip(*got):
        assert np.max(np.abs(x - y)) <= 1e-11 * np.max(np.abs(y))
