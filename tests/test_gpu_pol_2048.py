"""The polarised transforms at Nside 2048, where the spin-2 analysis takes its ring pairs in two launches: the
double-float form against the native one (bar 1e-11 of the largest output, as at the smaller sizes), and the analysis
as the adjoint of the synthesis, whose kernels take all ring pairs at once."""
import numpy as np
import pytest

from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


def test_analysis_is_the_adjoint_of_the_synthesis():
    import torch
    nside, lmax = 2048, 5
    npix, nalm = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    g = torch.Generator("cuda").manual_seed(1)
    a = torch.randn(3, nalm, 2, generator=g, device="cuda", dtype=torch.float64)
    a[:, :lmax + 1, 1] = 0.0
    below2 = np.concatenate([np.arange(m, lmax + 1) < 2 for m in range(lmax + 1)])
    a[1:, torch.from_numpy(below2).cuda()] = 0.0          # E and B begin at l = 2
    a = torch.view_as_complex(a)
    f = torch.randn(3, npix, generator=g, device="cuda", dtype=torch.float64)
    got = []
    for prec in (wf.WF_PREC_FP64, wf.WF_PREC_FP64_NATIVE):
        P = wf.Pol(nside, lmax, [np.ones(lmax + 1)] * 3 + [np.zeros(lmax + 1)],
                   np.tile([1.0, 1.0, 0.0, 1.0], (npix, 1)), opts=wf.options(precision=prec))
        m, t = torch.zeros_like(f), torch.zeros_like(a)
        torch.cuda.synchronize()
        P.alm2map(a.data_ptr(), m.data_ptr())
        torch.cuda.synchronize()
        f += m                                            # as large along Y a as across it
        torch.cuda.synchronize()
        P.map2alm(f.data_ptr(), t.data_ptr())
        torch.cuda.synchronize()
        P.close()
        wgt = torch.full((nalm,), 2.0, dtype=torch.float64, device="cuda")
        wgt[:lmax + 1] = 1.0
        for c in (slice(0, 1), slice(1, 3)):
            one = 4 * np.pi / npix * float((f[c] * m[c]).sum())
            other = float((wgt * (a[c].conj() * t[c]).real).sum())
            assert abs(one - other) <= 1e-11 * abs(one)
        f -= m
        got.append((m, t))
    for x, y in zip(*got):
        assert float((x - y).abs().max()) <= 1e-11 * float(y.abs().max())
