"""The recurrence form of the Legendre stage at the edges of its kernels against
the native FP64 form: ring pairs that fill part of a warp, of a thread's four or
of a chunk, band limits next to the blocks of 8 l, start values inside a block,
and both sides of the line between the smaller and the larger CTAs (RP = 2048).
Bar 1e-10 relative L2, the FP64 paths' parity bar."""
import numpy as np
import pytest

from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,lsht", [(1, 4, 3), (4, 9, 7), (8, 8, 8), (16, 47, 39), (32, 128, 121),
                                             (128, 300, 255), (512, 90, 88), (1024, 61, 57), (2048, 33, 33)])
def test_recurrence_against_native(nside, lmax, lsht):
    import torch
    npix, nalm = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    rng = np.random.default_rng(nside + lmax)
    a = rng.standard_normal(nalm) + 1j * rng.standard_normal(nalm)
    a[:lmax + 1].imag = 0.0
    f = rng.standard_normal(npix)
    cl = 1.0 / (1.0 + np.arange(lmax + 1)) ** 2
    got = []
    for kw in (dict(legendre_table_bytes=0), dict(precision=wf.WF_PREC_FP64_NATIVE)):
        P = wf.Plan(nside, lmax, cl, np.ones(npix), opts=wf.options(**kw))
        assert P.legendre_table(lmax)[0] == 0
        ad, fd = torch.from_numpy(a).cuda(), torch.from_numpy(f).cuda()
        m = torch.zeros(npix, dtype=torch.float64, device="cuda")
        t = torch.zeros(nalm, dtype=torch.complex128, device="cuda")
        s = torch.zeros(nalm, dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        P.alm2map(lsht, ad.data_ptr(), m.data_ptr())
        P.map2alm(lsht, fd.data_ptr(), t.data_ptr())
        P.iterate(fd.data_ptr(), s.data_ptr(), 2.0, lsht, 2)
        torch.cuda.synchronize()
        got.append([x.cpu().numpy() for x in (m, t, s)])
        P.close()
    for x, y in zip(*got):
        assert np.linalg.norm(x - y) <= 1e-10 * np.linalg.norm(y)
