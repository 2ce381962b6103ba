"""wf_map2alm_noalloc at the edges of its range: the smallest grids (a belt of
one length, rings with no, one and several Bluestein lengths), ring pairs that
fill part of a warp or of the block, and lmax from 0 up to 4 nside, where its
closed-form table offsets and its start values have their special cases. Bars
as for the other sizes: 1e-12 of the largest coefficient against the oracle,
1e-14 against a plan of the native FP64 kernels."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1211_0585_gb300 import wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax", [(1, 0), (1, 4), (2, 7), (4, 16), (8, 31), (32, 128), (64, 256), (128, 3),
                                        (128, 301)])
def test_noalloc_edges(nside, lmax):
    import torch
    rng = np.random.default_rng(1000 * nside + lmax)
    f_host = rng.standard_normal(12 * nside * nside)
    nalm = (lmax + 1) * (lmax + 2) // 2
    f = torch.from_numpy(f_host).cuda()
    got = torch.full((2 * nalm,), 3.0, dtype=torch.float64, device="cuda")
    wf.map2alm_noalloc(nside, lmax, f.data_ptr(), got.data_ptr())
    P = wf.Plan(nside, lmax, np.ones(lmax + 1), np.ones(f_host.size),
                opts=wf.options(precision=wf.WF_PREC_FP64_NATIVE))
    ref = torch.zeros_like(got)
    P.map2alm(lmax, f.data_ptr(), ref.data_ptr())
    torch.cuda.synchronize()
    P.close()
    g, r = got.cpu().numpy(), ref.cpu().numpy()
    assert np.max(np.abs(g - r)) <= 1e-14 * np.max(np.abs(r))
    orc = O.map2alm(nside, lmax, f_host).view(np.float64)
    assert np.max(np.abs(g - orc)) <= 1e-12 * np.max(np.abs(orc))
