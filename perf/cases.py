"""Timed cases of the messenger-field Wiener filter: the transforms, the iteration and the whole solves that a
program runs through paper_1211_0585_gb300.wf, from the smallest configuration (Nside 16, lmax 32) to the Planck-shaped
one (Nside 2048, lmax 4096).

Inputs are WMAP/Planck-shaped (the spectra, hit patterns, masks and noise levels of paper_1211_0585_gb300.inputs),
made on the GPU from the seed alone. `exact` evaluates the same quantities in float64 with plain torch: a Legendre
recurrence, matrix products over l or over ring pairs, and chirp-z ring transforms.
"""
import math

import numpy as np
import torch

from paper_1211_0585_gb300 import inputs, wf

DEV = "cuda"
F8, C16 = torch.float64, torch.complex128
EXACT_TABLE = 20e9     # bytes of one dense float64 [m, l, ring pair] table that exact() may hold


# ---------------------------------------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest configuration (Nside 16 / lmax 32), cooled, to 1e-4: hundreds of iterations of a few kernels of
        # a few microseconds, so launches and latencies are what counts
        dict(name="solve_16", kind="solve", nside=16, lmax=32, tol=1e-4, nominal=500),
        # the plan-free, allocation-free analysis that latency-critical callers use, at a size its scratch admits
        dict(name="noalloc_64", kind="noalloc", nside=64, lmax=128),
        # one synthesis of the WMAP-shaped problem (mock skies, the transform back)
        dict(name="synthesis_512", kind="synthesis", nside=512, lmax=1024, lsht=1024),
        # one analysis at a medium size with an odd lmax that is no multiple of any tile
        dict(name="analysis_256", kind="analysis", nside=256, lmax=667, lsht=667),
        # the headline: the WMAP-shaped filter, cooled, FP64, to a relative increment of 1e-6
        dict(name="solve_512", kind="solve", nside=512, lmax=1024, tol=1e-6, nominal=351),
        # the Planck-shaped problem: one full-band iteration; lambda_lm does not fit a table here
        dict(name="iterate_2048", kind="iterate", nside=2048, lmax=4096, lsht=4096, lam=1.0, niter=1),
        # 64 maps that share mask and noise through the mixed engine: 40 steps of the cooled solve (a capped run)
        dict(name="mixed_512x64", kind="batch", precision="mixed", nside=512, lmax=1024, nrhs=64, tol=1e-6,
             max_iter=40, nominal=40),
        # a few maps solved in FP64 together, an odd number of them, at a serving shape
        dict(name="fp64_256x5", kind="batch", precision="fp64", nside=256, lmax=512, nrhs=5, tol=1e-4, max_iter=10000,
             nominal=60),
        # constrained realisations: 7 draws and the Wiener filter of the data, host arrays in and out. In FP64: the
        # draws pass through a transform before the solves, and the FP32 steps of a mixed solve would turn a change in
        # that transform's last bit into another rounding everywhere
        dict(name="realisations_256x7", kind="realisations", nside=256, lmax=512, nreal=7, tol=1e-4, nominal=60),
        # three detectors with their own beams, noise and masks, joint filter
        dict(name="multi_256x3", kind="multi", nside=256, lmax=512, ndet=3, tol=1e-4, nominal=60),
        # temperature and polarisation, cooled joint filter at a serving shape
        dict(name="pol_solve_128", kind="pol_solve", nside=128, lmax=256, tol=1e-5, nominal=100),
        # the polarised transform pair of the WMAP-shaped problem
        dict(name="pol_pair_512", kind="pol_pair", nside=512, lmax=1024),
    ]


def _odd_lmax(rng, nside):
    return rng.randint(nside, 5 * nside // 2)


def draw(rng):
    kind = rng.choice(["solve", "noalloc", "synthesis", "analysis", "iterate", "batch", "realisations", "multi",
                       "pol_solve", "pol_pair"])
    if kind == "solve":
        ns = 2 ** rng.randint(3, 8)
        tol = 10.0 ** (rng.uniform(-6, -4) if ns > 32 else rng.uniform(-4, -3))
        return dict(kind=kind, nside=ns, lmax=_odd_lmax(rng, ns), tol=tol, nominal=200)
    if kind == "noalloc":
        ns = 2 ** rng.randint(2, 7)
        return dict(kind=kind, nside=ns, lmax=_odd_lmax(rng, ns))
    if kind in ("synthesis", "analysis"):
        ns = 2 ** rng.randint(4, 10)
        lmax = _odd_lmax(rng, ns)
        return dict(kind=kind, nside=ns, lmax=lmax, lsht=lmax if rng.random() < 0.5 else rng.randint(lmax // 4, lmax))
    if kind == "iterate":
        ns = 2 ** rng.randint(4, 10)
        lmax = _odd_lmax(rng, ns)
        return dict(kind=kind, nside=ns, lmax=lmax, lsht=lmax if rng.random() < 0.5 else rng.randint(lmax // 4, lmax),
                    lam=rng.choice([1.0, 3.0, 40.0]), niter=rng.randint(1, 6))
    if kind == "batch":
        ns = 2 ** rng.randint(4, 8)
        return dict(kind=kind, precision=rng.choice(["mixed", "fp64"]), nside=ns, lmax=_odd_lmax(rng, ns),
                    nrhs=rng.randint(2, 40 if ns < 256 else 12), tol=1e-4, max_iter=10000, nominal=60)
    if kind == "realisations":
        ns = 2 ** rng.randint(4, 8)
        return dict(kind=kind, nside=ns, lmax=_odd_lmax(rng, ns), nreal=rng.randint(1, 7), tol=1e-4, nominal=60)
    if kind == "multi":
        ns = 2 ** rng.randint(3, 8)
        return dict(kind=kind, nside=ns, lmax=_odd_lmax(rng, ns), ndet=rng.randint(2, 5), tol=1e-4, nominal=60)
    if kind == "pol_solve":
        ns = 2 ** rng.randint(3, 7)
        return dict(kind=kind, nside=ns, lmax=_odd_lmax(rng, ns), tol=1e-4, nominal=80)
    ns = 2 ** rng.randint(4, 9)
    return dict(kind=kind, nside=ns, lmax=rng.randint(ns, 2 * ns))


def work(case):
    """Inputs read once and outputs written once; the flops of the transforms: a Legendre sum over every (l, m, ring
    pair) (4 real multiply-adds: two parities share the pair's two rings) and a real FFT of every ring."""
    ns, lmax, kind = case["nside"], case["lmax"], case["kind"]
    L = case.get("lsht", lmax)
    npix, nalm = 12 * ns * ns, (lmax + 1) * (lmax + 2) // 2
    ltri = (L + 1) * (L + 2) // 2
    sht = 8.0 * ltri * 2 * ns + 2.5 * npix * math.log2(4 * ns)
    pix, alm = 8 * npix, 16 * nalm
    if kind in ("noalloc", "synthesis", "analysis"):
        return dict(bytes=pix + 16 * ltri, flops=sht)
    if kind == "iterate":
        return dict(bytes=2 * pix + 2 * alm, flops=2 * sht * case["niter"])
    it = case.get("nominal", 1)
    if kind == "solve":
        return dict(bytes=2 * pix + alm, flops=2 * sht * it)
    if kind == "batch":
        return dict(bytes=pix + case["nrhs"] * (pix + alm), flops=2 * sht * it * case["nrhs"])
    if kind == "realisations":
        n = case["nreal"] + 1
        return dict(bytes=2 * pix + n * alm, flops=2 * sht * it * n)
    if kind == "multi":
        return dict(bytes=case["ndet"] * 2 * pix + alm, flops=2 * sht * it * case["ndet"])
    pol = 8.0 * 4 * ltri * 2 * ns + 2 * 2.5 * npix * math.log2(4 * ns) + sht   # spin 2: F+ and F- on two fields
    if kind == "pol_solve":
        return dict(bytes=3 * pix + 4 * pix + 3 * alm, flops=2 * pol * it)
    return dict(bytes=2 * 3 * (pix + alm), flops=2 * pol)


# --------------------------------------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(DEV).manual_seed(seed)


def _sky(nside, seed):
    """(z, phi, unit vectors, generator) of the pixels."""
    z, phi = inputs.pixel_centres(nside)
    z, phi = torch.from_numpy(z).to(DEV), torch.from_numpy(phi).to(DEV)
    s = torch.sqrt(torch.clamp(1 - z * z, min=0))
    return z, torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], 1).float(), _gen(seed)


def _cl(nside, lmax):
    if nside <= 32:
        return inputs.cl_inverse_square(lmax)
    return inputs.cl_lcdm_like(lmax, 13.0 if nside <= 512 else 5.0)


def _hits(v):
    sb = v[:, 0].double() * math.sin(math.radians(60.0)) + v[:, 2].double() * math.cos(math.radians(60.0))
    return sb.abs()


def _noise(nside, v, cl):
    if nside <= 32:
        return 1e-3 * float(cl[2]) / (1 + 2 * _hits(v))
    return 2200.0 ** 2 * (nside / 512) ** 2 / (1 + 7 * _hits(v))


def _mask(z, v, g, band, discs):
    """A band cut about the equator and discs of half a degree."""
    m = z.abs() >= band
    if discs:
        c = torch.nn.functional.normalize(torch.randn(discs, 3, generator=g, device=DEV), dim=1)
        for a in range(0, v.shape[0], 1 << 20):
            m[a:a + (1 << 20)] &= ~((v[a:a + (1 << 20)] @ c.T).amax(1) > math.cos(math.radians(0.5)))
    return m


def _signal(v, cl, g, n=1):
    """n Gaussian-like random skies [n, npix] of power C_l: plane waves of wave number l + 1/2, with random
    directions, phases and amplitudes, (2 l + 1) C_l / 4 pi of variance each band of l (to 0.7 lmax where the noise is
    far below the signal: a wave reaches a little beyond its own l)."""
    top = len(cl) if len(cl) > 100 else max(4, int(0.7 * len(cl)))
    l = torch.arange(2, top, device=DEV, dtype=F8)
    c = torch.as_tensor(cl, device=DEV)[2:top]
    var = (2 * l + 1) * c / (4 * math.pi)
    J = 192
    pick = torch.multinomial((2 * l + 1) * c, J, replacement=True, generator=g)
    k = torch.nn.functional.normalize(torch.randn(J, 3, generator=g, device=DEV), dim=1) * (l[pick].float() + 0.5)[:, None]
    ph = 2 * math.pi * torch.rand(J, generator=g, device=DEV)
    amp = torch.randn(J, n, generator=g, device=DEV) * math.sqrt(2 * float(var.sum()) / J)
    out = torch.empty(n, v.shape[0], dtype=F8, device=DEV)
    for a in range(0, v.shape[0], 1 << 20):
        out[:, a:a + (1 << 20)] = (torch.cos(v[a:a + (1 << 20)] @ k.T + ph) @ amp).T.double()
    low = torch.cat([torch.ones_like(v[:, :1]), math.sqrt(3.0) * v], 1).double()   # C_0 = C_1 = 0
    return out.sub_((out @ low) @ low.T / v.shape[0])


def _alm(cl, g):
    """a_lm ~ N(0, C_l), m >= 0, m-major."""
    ls, ms = inputs.alm_lm_arrays(len(cl) - 1)
    var = torch.as_tensor(cl, device=DEV)[torch.from_numpy(ls).to(DEV)]
    m0 = torch.from_numpy(ms).to(DEV) == 0
    re = torch.randn(var.numel(), generator=g, device=DEV, dtype=F8)
    im = torch.randn(var.numel(), generator=g, device=DEV, dtype=F8)
    sd = torch.sqrt(torch.where(m0, var, var / 2))
    return torch.complex(re * sd, torch.where(m0, 0.0, im * sd))


def _problem(case, seed, nmaps=1):
    """C_l, noise variance, mask and data [nmaps, npix] of a temperature problem, on the GPU."""
    ns, lmax = case["nside"], case["lmax"]
    z, v, g = _sky(ns, seed)
    cl = _cl(ns, lmax)
    nv = _noise(ns, v, cl)
    mask = _mask(z, v, g, math.sin(math.radians(10.0)) if ns <= 32 else 0.2, 0 if ns <= 32 or ns > 512 else 500)
    d = _signal(v, cl, g, nmaps)
    for i in range(nmaps):
        d[i] += torch.sqrt(nv) * torch.randn(d.shape[1], generator=g, device=DEV, dtype=F8)
    return cl, nv, mask, d


def _inputs(case, seed):
    """Every array the case's call needs."""
    ns, lmax, kind = case["nside"], case["lmax"], case["kind"]
    if kind in ("solve", "iterate"):
        cl, nv, mask, d = _problem(case, seed)
        return dict(cl=cl, nv=nv, mask=mask, d=d[0])
    if kind == "batch":
        cl, nv, mask, d = _problem(case, seed, case["nrhs"])
        return dict(cl=cl, nv=nv, mask=mask, d=d)
    if kind == "realisations":
        cl, nv, mask, d = _problem(case, seed)
        return dict(cl=cl, nv=nv, mask=mask, d=d[0], seed=seed)
    if kind == "multi":
        K = case["ndet"]
        z, v, g = _sky(ns, seed)
        cl = _cl(ns, lmax)
        sky = _signal(v, cl, g)[0]
        nv, mask, d = [], [], []
        for k in range(K):
            nv.append(_noise(ns, v, cl) * (1 + 0.5 * k))
            mask.append(_mask(z, v, g, 0.1 + 0.05 * k, 0 if ns <= 32 else 100))
            d.append(sky + torch.sqrt(nv[k]) * torch.randn(sky.numel(), generator=g, device=DEV, dtype=F8))
        fwhm = 3000.0 / ns
        return dict(cl=cl, nv=torch.stack(nv), mask=torch.stack(mask), d=torch.stack(d),
                    beams=np.stack([inputs.gaussian_beam(lmax, fwhm * (1 + k)) for k in range(K)]))
    if kind in ("pol_solve", "pol_pair"):
        z, v, g = _sky(ns, seed)
        tt = _cl(ns, lmax)
        cls = np.stack([tt, tt / 30, tt / 1000, 0.3 * np.sqrt(tt * tt / 30)])
        if kind == "pol_pair":
            return dict(cls=cls, alm=torch.stack([_alm(cls[i], g) for i in range(3)]))
        cov = torch.zeros(z.numel(), 4, dtype=F8, device=DEV)
        cov[:, 0] = _noise(ns, v, tt)
        cov[:, 1] = cov[:, 3] = 2 * cov[:, 0]
        cov[:, 2] = 0.2 * cov[:, 1] * (2 * torch.rand(z.numel(), generator=g, device=DEV, dtype=F8) - 1)
        mt = _mask(z, v, g, 0.2, 0 if ns <= 32 else 200)
        mp = mt & (z.abs() >= 0.3)
        e = torch.randn(3, z.numel(), generator=g, device=DEV, dtype=F8)
        l11 = torch.sqrt(cov[:, 1])
        l21 = cov[:, 2] / l11
        d = torch.stack([_signal(v, cls[i], g)[0] for i in (0, 1, 1)])
        d += torch.stack([torch.sqrt(cov[:, 0]) * e[0], l11 * e[1], l21 * e[1] + torch.sqrt(cov[:, 3] - l21 ** 2) * e[2]])
        return dict(cls=cls, nv=cov, mask_t=mt, mask_p=mp, d=d)
    cl = _cl(ns, lmax)
    if kind == "synthesis":
        return dict(cl=cl, alm=_alm(cl, _gen(seed)))
    _, v, g = _sky(ns, seed)
    d = _signal(v, cl, g)[0]
    return dict(cl=cl, map=d + torch.randn(d.numel(), generator=g, device=DEV, dtype=F8) * d.std())


def _host(t):
    return t.cpu().numpy()


# ------------------------------------------------------------------------------------------------------ the calls

def prepare(case, seed):
    ns, lmax, kind = case["nside"], case["lmax"], case["kind"]
    q = _inputs(case, seed)
    npix, nalm = 12 * ns * ns, (lmax + 1) * (lmax + 2) // 2
    s = dict(case=case)
    if kind == "noalloc":
        s.update(map=q["map"], out=torch.zeros(nalm, dtype=C16, device=DEV))
    elif kind in ("synthesis", "analysis"):
        s["plan"] = wf.Plan(ns, lmax, q["cl"], np.ones(npix))
        if kind == "synthesis":
            s.update(alm=q["alm"], out=torch.zeros(npix, dtype=F8, device=DEV))
        else:
            s.update(map=q["map"], out=torch.zeros(nalm, dtype=C16, device=DEV))
    elif kind in ("solve", "iterate"):
        opts = wf.options(tol=case.get("tol", 1e-6))
        s.update(plan=wf.Plan(ns, lmax, q["cl"], _host(q["nv"]), _host(q["mask"]), opts), d=q["d"],
                 out=torch.zeros(nalm, dtype=C16, device=DEV))
        if kind == "iterate":   # from a state with the signal's power in every mode of the band
            ls, _ = inputs.alm_lm_arrays(lmax)
            s["start"] = _alm(q["cl"], _gen(seed + 1)) * torch.from_numpy(ls <= case["lsht"]).to(DEV)
    elif kind == "batch":
        p = wf.WF_PREC_MIXED if case["precision"] == "mixed" else wf.WF_PREC_FP64
        opts = wf.options(precision=p, tol=case["tol"], max_iter=case["max_iter"], batch_slots=case["nrhs"])
        s.update(plan=wf.Plan(ns, lmax, q["cl"], _host(q["nv"]), _host(q["mask"]), opts), d=q["d"],
                 out=torch.zeros(case["nrhs"], nalm, dtype=C16, device=DEV))
    elif kind == "realisations":
        opts = wf.options(tol=case["tol"])
        s.update(plan=wf.Plan(ns, lmax, q["cl"], _host(q["nv"]), _host(q["mask"]), opts), d=_host(q["d"]), seed=q["seed"])
    elif kind == "multi":
        s.update(plan=wf.Multi(ns, lmax, q["cl"], list(_host(q["nv"])), list(_host(q["mask"])), list(q["beams"]),
                               wf.options(tol=case["tol"])), d=_host(q["d"]))
    elif kind == "pol_solve":
        s.update(plan=wf.Pol(ns, lmax, list(q["cls"]), _host(q["nv"]), _host(q["mask_t"]), _host(q["mask_p"]),
                             wf.options(tol=case["tol"])), d=_host(q["d"]))
    else:
        noise = np.tile([1.0, 2.0, 0.0, 2.0], (npix, 1))
        s.update(plan=wf.Pol(ns, lmax, list(q["cls"]), noise), alm=q["alm"],
                 map=torch.zeros(3, npix, dtype=F8, device=DEV), out=torch.zeros(3, nalm, dtype=C16, device=DEV))
    torch.cuda.synchronize()   # the plan runs on a stream of its own
    return s


def _told(st):
    """The figures of a solve that a program reads: how many iterations and the chi^2 they ended with."""
    return dict(iters=st["iters"], levels=st["levels"], chi2_prior=st["chi2_prior"], chi2_noise=st["chi2_noise"])


def run(s):
    c = s["case"]
    kind, plan = c["kind"], s.get("plan")
    if kind == "noalloc":
        wf.map2alm_noalloc(c["nside"], c["lmax"], s["map"].data_ptr(), s["out"].data_ptr())
        return s["out"]
    if kind == "synthesis":
        plan.alm2map(c["lsht"], s["alm"].data_ptr(), s["out"].data_ptr())
        return s["out"]
    if kind == "analysis":
        plan.map2alm(c["lsht"], s["map"].data_ptr(), s["out"].data_ptr())
        return s["out"]
    if kind == "iterate":
        s["out"].copy_(s["start"])
        torch.cuda.current_stream().synchronize()   # the state in place before the plan's own stream reads it
        recs = plan.iterate(s["d"].data_ptr(), s["out"].data_ptr(), c["lam"], c["lsht"], c["niter"])
        return dict(alm=s["out"], chi2=np.array([r["chi2"] for r in recs]), norm2=np.array([r["norm2"] for r in recs]))
    if kind == "solve":
        _, st, _, _ = plan.solve(s["d"].data_ptr(), s["out"].data_ptr(), on_device=True)
        return dict(alm=s["out"], **_told(st))
    if kind == "batch":
        _, st, _ = plan.solve_batch(s["d"].data_ptr(), on_device=True, alm_out=s["out"].data_ptr(), nrhs=c["nrhs"])
        return dict(alm=s["out"], iters=np.array([x["iters"] for x in st]), chi2=np.array([x["chi2"] for x in st]))
    if kind == "realisations":
        cr, wfm, st, _ = plan.constrained_realisations(s["d"], c["nreal"], s["seed"])
        return dict(cr=cr, wf=wfm, iters=np.array([x["iters"] for x in st]))
    if kind in ("multi", "pol_solve"):
        alm, st, _, _ = plan.solve(s["d"])
        return dict(alm=alm, **_told(st))
    plan.alm2map(s["alm"].data_ptr(), s["map"].data_ptr())
    plan.map2alm(s["map"].data_ptr(), s["out"].data_ptr())
    return dict(map=s["map"], alm=s["out"])


# ----------------------------------------------------------------------------------------- the same in plain float64

class Sht:
    """Spherical-harmonic synthesis and its adjoint on a HEALPix grid in float64, on [m, l] arrays of coefficients."""

    def __init__(self, nside, lmax, spin2=False, table=True):
        self.ns, self.L = nside, lmax
        self.npix = 12 * nside * nside
        self.omega = 4 * math.pi / self.npix
        R = self.R = 4 * nside - 1
        i = torch.arange(1, R + 1, device=DEV)
        ip = torch.minimum(i, 4 * nside - i)
        cap = ip < nside
        self.n = torch.where(cap, 4 * ip, 4 * nside)
        shifted = cap | ((i - nside) % 2 == 0)
        self.phi0 = torch.where(shifted, math.pi / self.n.to(F8), 0.0)
        zi = i[:2 * nside].to(F8)
        self.x = torch.where(cap[:2 * nside], 1 - zi * zi / (3.0 * nside ** 2), 4.0 / 3 - 2 * zi / (3.0 * nside))
        self.sn2 = torch.where(cap[:2 * nside], zi * zi / (3.0 * nside ** 2) * (2 - zi * zi / (3.0 * nside ** 2)),
                               (1 - self.x) * (1 + self.x))
        # chirp-z ring transforms: w_j = e^{i pi j^2 / n}
        N = 4 * nside
        self.M = 1 << (2 * N - 1).bit_length()
        j = torch.arange(N, device=DEV)
        n = self.n[:, None]
        self.w = torch.polar(torch.ones((), dtype=F8, device=DEV), math.pi * ((j * j) % (2 * n)).to(F8) / n) * (j < n)
        self.inside = j < n
        m = torch.arange(lmax + 1, device=DEV)
        self.q = m % n                                             # [R, m]
        self.em = torch.polar(torch.ones((), dtype=F8, device=DEV), torch.remainder(m * self.phi0[:, None], 2 * math.pi))
        self.sgn = 1.0 - 2.0 * ((m[None, :] - m[:, None]) % 2).to(F8)   # (-1)^(l - m) [m, l]
        ls, ms = inputs.alm_lm_arrays(lmax)
        self.at = (torch.from_numpy(ms).to(DEV), torch.from_numpy(ls).to(DEV))
        if table:
            self.T = torch.empty(lmax + 1, lmax + 1, 2 * nside, dtype=F8, device=DEV)
            if spin2:
                self.FP, self.FM = torch.zeros_like(self.T), torch.zeros_like(self.T)
            last = None
            for l, lam in self.rows():
                self.T[:, l] = lam
                if spin2 and l >= 2:
                    mm = m[:, None].to(F8)
                    nl = 1 / math.sqrt((l - 1.0) * l * (l + 1) * (l + 2))
                    c = torch.sqrt(torch.clamp((2 * l + 1) / (2 * l - 1.0) * (l * l - mm * mm), min=0)) * last
                    self.FP[:, l] = nl * ((2 * (mm * mm - l) / self.sn2 - l * (l - 1.0)) * lam + 2 * self.x * c / self.sn2)
                    self.FM[:, l] = nl * 2 * mm / self.sn2 * (c - (l - 1.0) * self.x * lam)
                    self.FP[l + 1:, l] = 0
                    self.FM[l + 1:, l] = 0
                last = lam

    def rows(self):
        """(l, lambda_lm at the northern rings [m, ring pair], zero for m > l), l ascending; every column carries an
        exponent of its own, brought up to date every 16 steps."""
        L, x = self.L, self.x
        m = torch.arange(L + 1, device=DEV, dtype=F8)[:, None]
        mant = torch.zeros(L + 1, x.numel(), dtype=F8, device=DEV)
        # lambda_mm = (-1)^m sqrt((2m+1)/4pi prod (2i-1)/2i) sin^m: mantissa and power of two by repeated products
        v = torch.full_like(x, 1 / math.sqrt(4 * math.pi))
        e = torch.zeros_like(x)
        start, sexp = torch.empty_like(mant), torch.empty_like(mant)
        sth = torch.sqrt(self.sn2)
        for k in range(L + 1):
            if k:
                v = -v * math.sqrt((2 * k + 1) / (2.0 * k)) * sth
                f, ex = torch.frexp(v)
                v, e = f, e + ex
            start[k], sexp[k] = v, e
        p1, p2 = torch.zeros_like(mant), mant
        exp = sexp
        scale = torch.exp2(torch.clamp(exp, min=-1080))
        for l in range(L + 1):
            a = torch.sqrt((4.0 * l * l - 1) / torch.clamp(l * l - m * m, min=1)) if l else torch.zeros_like(m)
            b = a * torch.sqrt(torch.clamp((l - 1.0) ** 2 - m * m, min=0) / max(4.0 * (l - 1) ** 2 - 1, 1.0))
            new = a * x * p1 - b * p2
            new[l] = start[l]
            new[l + 1:] = 0
            p2, p1 = p1, new
            if l % 16 == 15:
                _, ex = torch.frexp(torch.maximum(p1.abs(), p2.abs()))
                p1, p2 = torch.ldexp(p1, -ex), torch.ldexp(p2, -ex)
                exp = exp + ex
                scale = torch.exp2(torch.clamp(exp, min=-1080))
            yield l, p1 * scale

    def dense(self, alm):
        out = torch.zeros(*alm.shape[:-1], self.L + 1, self.L + 1, dtype=C16, device=DEV)
        out[(..., *self.at)] = alm
        return out

    def packed(self, A):
        return A[(..., *self.at)]

    # Legendre sums: A [B, m, l] <-> coefficients of every ring [B, R, m]
    def _up(self, tab, A):
        v = torch.view_as_real(A).permute(1, 0, 3, 2)                      # [m, B, 2, l]
        B = v.shape[1]
        v = torch.cat([v, v * self.sgn[:, None, None, :]], 1).reshape(self.L + 1, 4 * B, self.L + 1)
        f = torch.bmm(v, tab).reshape(self.L + 1, 2, B, 2, -1).permute(1, 2, 4, 0, 3).contiguous()
        return torch.view_as_complex(f)                                    # [north / south, B, pair, m]

    def _down(self, tab, F):
        v = torch.view_as_real(F).permute(3, 2, 0, 1, 4)                   # [m, pair, ns, B, 2]
        B = v.shape[3]
        t = torch.bmm(tab, v.reshape(self.L + 1, v.shape[1], 4 * B)).reshape(self.L + 1, self.L + 1, 2, B, 2)
        t = t[:, :, 0] + self.sgn[:, :, None, None] * t[:, :, 1]
        return torch.view_as_complex(t.permute(2, 0, 1, 3).contiguous())   # [B, m, l]

    def _rings(self, F):
        return torch.cat([F[0], F[1][:, :-1].flip(1)], 1)                  # [B, R, m]

    def _pairs(self, U):
        n, s = U[:, :2 * self.ns], torch.zeros_like(U[:, :2 * self.ns])
        s[:, :-1] = U[:, 2 * self.ns:].flip(1)
        return torch.stack([n, s])

    def _chirp(self, v, w):
        """sum_q v_q e^{+-2 pi i q p / n} on every ring: v [.., R, N], w the chirp or its conjugate."""
        b = torch.zeros(self.R, self.M, dtype=C16, device=DEV)
        N = self.w.shape[1]
        b[:, :N] = w.conj()
        b[:, self.M - N + 1:] = w[:, 1:].conj().flip(1)
        y = torch.fft.ifft(torch.fft.fft(v * w, self.M) * torch.fft.fft(b))
        return y[..., :N] * w

    def to_map(self, F):
        """F [B, R, m] -> maps [B, npix]."""
        out = torch.empty(F.shape[0], self.npix, dtype=F8, device=DEV)
        for b in range(F.shape[0]):
            c = F[b] * self.em
            c[:, 1:] *= 2
            G = torch.zeros(self.R, self.w.shape[1], 2, dtype=F8, device=DEV)
            G.scatter_add_(1, self.q[..., None].expand(-1, -1, 2), torch.view_as_real(c))
            out[b] = self._chirp(torch.view_as_complex(G), self.w).real[self.inside]   # RING order
        return out

    def from_map(self, maps):
        """maps [B, npix] -> Omega sum_p u_p e^{-i m phi_p} of every ring [B, R, m]."""
        out = torch.empty(maps.shape[0], self.R, self.L + 1, dtype=C16, device=DEV)
        for b in range(maps.shape[0]):
            u = torch.zeros(self.R, self.w.shape[1], dtype=C16, device=DEV)
            u[self.inside] = maps[b].to(C16)
            out[b] = self.omega * torch.gather(self._chirp(u, self.w.conj()), 1, self.q) * self.em.conj()
        return out

    def synthesis(self, A):
        return self.to_map(self._rings(self._up(self.T, A)))

    def analysis(self, maps):
        return self._down(self.T, self._pairs(self.from_map(maps)))

    def synthesis_rows(self, A):
        """As synthesis, the Legendre functions generated row by row instead of held."""
        n = torch.zeros(2 * self.ns, self.L + 1, 2, dtype=F8, device=DEV).permute(2, 1, 0).contiguous()   # [2, m, pair]
        s = torch.zeros_like(n)
        for l, lam in self.rows():
            a = torch.view_as_real(A[0, :l + 1, l])
            for c in range(2):
                n[c, :l + 1].addcmul_(lam[:l + 1], a[:, c:c + 1])
                s[c, :l + 1].addcmul_(lam[:l + 1], (a[:, c] * self.sgn[:l + 1, l])[:, None])
        F = torch.stack([torch.complex(v[0], v[1]).T for v in (n, s)])[:, None]
        return self.to_map(self._rings(F))

    def analysis_rows(self, maps):
        F = self._pairs(self.from_map(maps))[:, 0].permute(2, 1, 0)                # [m, pair, ns]
        even, odd = F[..., 0] + F[..., 1], F[..., 0] - F[..., 1]
        parts = [[x.real.contiguous(), x.imag.contiguous()] for x in (even, odd)]
        t = torch.zeros(1, self.L + 1, self.L + 1, 2, dtype=F8, device=DEV)
        for l, lam in self.rows():
            for c in range(2):
                for par in range(2):
                    at = slice((l + par) % 2, l + 1, 2)
                    t[0, at, l, c] = (lam[at] * parts[par][c][at]).sum(1)
        return torch.view_as_complex(t)

    # (E, B) [2, m, l] <-> (Q, U) [2, npix]; F- changes sign with the parity where F+ does not
    def synthesis2(self, EB):
        p, q = self._up(self.FP, EB), self._up(self.FM, EB)
        flip = torch.tensor([1.0, -1.0], dtype=F8, device=DEV)[:, None, None]
        Q = -(p[:, 0] + 1j * q[:, 1] * flip)
        U = -(p[:, 1] - 1j * q[:, 0] * flip)
        return self.to_map(self._rings(torch.stack([Q, U], 1)))

    def analysis2(self, QU):
        F = self._pairs(self.from_map(QU))
        flip = torch.tensor([1.0, -1.0], dtype=F8, device=DEV)[:, None, None, None]
        p, q = self._down(self.FP, F), self._down(self.FM, F * flip)
        out = torch.stack([-(p[0] + 1j * q[1]), -(p[1] - 1j * q[0])])
        out[:, :, :2] = 0
        return out


def _cooled(lmax, lam_of, band, sigma, tol, step, max_iter=10000):
    """The cooling schedule and stop rule (defaults of wf.options) about step(lambda, band limit), which advances the
    state and gives (chi2 prior, chi2 noise, ||increment||^2, ||state||^2). Returns (iterations, levels, last step)."""
    l_iter, level, since, prev, it = 20, 0, 0, None, 0
    lam = lam_of(20)
    lsht = lmax if lam <= 1 or not band else min(lmax, 120)
    while True:
        got = step(lam, lsht)
        it, since = it + 1, since + 1
        chi2 = got[0] + got[1]
        d = abs(chi2 - prev) if prev is not None and since >= 3 else None
        prev = chi2
        if lam > 1:
            if (d is not None and d < 1e-2 * sigma) or since >= 1000:
                l_iter *= 2
                lam, level, since, prev = min(lam, lam_of(l_iter)), level + 1, 0, None
                lsht = lmax if lam <= 1 or not band else min(lmax, l_iter + 100)
        elif since >= 2 and got[2] <= tol ** 2 * got[3]:
            return it, level + 1, got
        if it >= max_iter:
            return it, level + 1, got


def _lam_of(cl, noise):
    return lambda l: 1.0 if l >= len(cl) else max(1.0, float(cl[l]) / noise)


def _filter(T, cl, nv, mask, d, tol=0.0, fixed=None, start=None, max_iter=10000, synth=None, ana=None):
    """One Wiener filter of one map; fixed = (lambda, band limit, iterations)."""
    synth, ana = synth or T.synthesis, ana or T.analysis
    w = torch.where(mask, 1 / nv, 0.0)
    tau = float(nv[mask].min())
    C = torch.as_tensor(cl, device=DEV)
    s = [torch.zeros(1, T.L + 1, T.L + 1, dtype=C16, device=DEV) if start is None else start]
    wm = torch.full((T.L + 1, 1), 2.0, dtype=F8, device=DEV)
    wm[0] = 1
    icl = torch.where(C > 0, 1 / C, 0.0)
    rec = []

    def sq(a, per_l=1.0):
        return float((wm * per_l * (a.real ** 2 + a.imag ** 2)).sum())

    def step(lam, lsht):
        a = s[0]
        r = d - synth(a)[0] if a.any() else d.clone()
        g = w / (1 + (lam - 1) * tau * w)
        t = ana((lam * tau * g * r)[None])
        new = (a + t) * (C / (C + lam * tau * T.omega))
        new[:, :, lsht + 1:] = 0
        got = sq(a, icl), float((w * r * r).sum()), sq(new - a), sq(new)
        s[0] = new
        rec.append(got)
        return got

    if fixed:
        for _ in range(fixed[2]):
            step(fixed[0], fixed[1])
        return T.packed(s[0])[0], rec
    it, levels, got = _cooled(T.L, _lam_of(cl, tau * T.omega), True, math.sqrt(2.0 * int(mask.sum())), tol, step, max_iter)
    return T.packed(s[0])[0], dict(iters=it, levels=levels, chi2_prior=got[0], chi2_noise=got[1])


def _joint(T, cl, q, tol):
    """The joint filter of several maps."""
    K = q["d"].shape[0]
    w = torch.where(q["mask"], 1 / q["nv"], 0.0)
    tau = torch.stack([q["nv"][k][q["mask"][k]].min() for k in range(K)])
    C, b = torch.as_tensor(cl, device=DEV), torch.as_tensor(q["beams"], device=DEV)
    wm = torch.full((T.L + 1, 1), 2.0, dtype=F8, device=DEV)
    wm[0] = 1
    icl = torch.where(C > 0, 1 / C, 0.0)
    s = [torch.zeros(T.L + 1, T.L + 1, dtype=C16, device=DEV)]

    def sq(a, per_l=1.0):
        return float((wm * per_l * (a.real ** 2 + a.imag ** 2)).sum())

    def step(lam, lsht):
        a = s[0]
        r = q["d"] - T.synthesis(a[None] * b[:, None, :])
        g = w / (1 + (lam - 1) * tau[:, None] * w)
        t = T.analysis(lam * tau[:, None] * g * r)
        gk = (1 / (lam * tau * T.omega))[:, None] * b
        new = (gk[:, None, :] * (b[:, None, :] * a + t)).sum(0) / torch.where(C > 0, 1 / C + (gk * b).sum(0), math.inf)
        got = sq(a, icl), float((w * r * r).sum()), sq(new - a), sq(new)
        s[0] = new
        return got

    comb = cl * _host((b * b / tau[:, None]).sum(0))
    it, levels, got = _cooled(T.L, _lam_of(comb, T.omega), False, math.sqrt(2.0 * int(q["mask"].sum())), tol, step)
    return dict(alm=T.packed(s[0]), iters=it, levels=levels, chi2_prior=got[0], chi2_noise=got[1])


def _polarised(T, q, tol):
    """The joint filter of (T, Q, U)."""
    cov = q["nv"]
    det = cov[:, 1] * cov[:, 3] - cov[:, 2] ** 2
    wt = torch.where(q["mask_t"], 1 / cov[:, 0], 0.0)
    w11, w12, w22 = (torch.where(q["mask_p"], x / det, 0.0) for x in (cov[:, 3], -cov[:, 2], cov[:, 1]))
    eig = 0.5 * (cov[:, 1] + cov[:, 3]) - torch.sqrt(0.25 * (cov[:, 1] - cov[:, 3]) ** 2 + cov[:, 2] ** 2)
    tau = min(float(cov[:, 0][q["mask_t"]].min()), float(eig[q["mask_p"]].min()))
    tt, ee, bb, te = torch.as_tensor(q["cls"], device=DEV)
    sdet = tt * ee - te * te
    wm = torch.full((T.L + 1, 1), 2.0, dtype=F8, device=DEV)
    wm[0] = 1
    s = [torch.zeros(3, T.L + 1, T.L + 1, dtype=C16, device=DEV)]

    def n2(a):
        return a.real ** 2 + a.imag ** 2

    def over(x, y):
        return torch.where(y > 0, x / torch.where(y > 0, y, 1.0), 0.0)

    def step(lam, lsht):
        a = s[0]
        m = torch.cat([T.synthesis(a[:1]), T.synthesis2(a[1:])])
        rt, rq, ru = q["d"] - m
        c, lt, k = (lam - 1) * tau, lam * tau, lam * tau * T.omega
        gt = wt / (1 + c * wt)
        a11, a12, a22 = 1 + c * w11, c * w12, 1 + c * w22
        dd = a11 * a22 - a12 * a12
        g11, g12, g22 = (w11 * a22 - w12 * a12) / dd, (w12 * a11 - w11 * a12) / dd, (w22 * a11 - w12 * a12) / dd
        t = a + torch.cat([T.analysis((lt * gt * rt)[None]),
                           T.analysis2(torch.stack([lt * (g11 * rq + g12 * ru), lt * (g12 * rq + g22 * ru)]))])
        de = (tt + k) * (ee + k) - te * te
        nT = ((tt * (ee + k) - te * te) * t[0] + te * k * t[1]) / de
        nE = (te * k * t[0] + (ee * (tt + k) - te * te) * t[1]) / de
        new = torch.stack([nT, nE, t[2] * over(bb, bb + k)])
        cross = a[0].real * a[1].real + a[0].imag * a[1].imag
        prior = torch.where(sdet > 0, over(ee * n2(a[0]) - 2 * te * cross + tt * n2(a[1]), sdet), over(n2(a[0]), tt))
        prior = prior + over(n2(a[2]), bb)
        noise = wt * rt * rt + w11 * rq * rq + 2 * w12 * rq * ru + w22 * ru * ru
        got = float((wm * prior).sum()), float(noise.sum()), float((wm * n2(new - a)).sum()), float((wm * n2(new)).sum())
        s[0] = new
        return got

    nobs = int(q["mask_t"].sum()) + 2 * int(q["mask_p"].sum())
    it, levels, got = _cooled(T.L, _lam_of(q["cls"][0], tau * T.omega), False, math.sqrt(2.0 * nobs), tol, step)
    return dict(alm=T.packed(s[0]), iters=it, levels=levels, chi2_prior=got[0], chi2_noise=got[1])


def exact(case, seed):
    ns, lmax, kind = case["nside"], case["lmax"], case["kind"]
    held = (lmax + 1) ** 2 * 2 * ns * 8 <= EXACT_TABLE
    if not held and kind not in ("synthesis", "analysis", "iterate", "noalloc"):
        return None
    maps = case.get("nrhs", 1)
    if kind == "batch" and work(case)["flops"] > 4e12:
        return None       # minutes of float64 matrix products
    q = _inputs(case, seed)
    T = Sht(ns, lmax, spin2=kind.startswith("pol"), table=held)
    synth, ana = (T.synthesis, T.analysis) if held else (T.synthesis_rows, T.analysis_rows)
    L = case.get("lsht", lmax)
    if kind == "synthesis":
        A = T.dense(q["alm"])[None]
        A[:, :, L + 1:] = 0
        return synth(A)[0]
    if kind in ("analysis", "noalloc"):
        A = ana(q["map"][None])
        A[:, :, L + 1:] = 0
        return T.packed(A)[0]
    if kind == "pol_pair":
        A = T.dense(q["alm"])
        m = torch.cat([T.synthesis(A[:1]), T.synthesis2(A[1:])])
        return dict(map=m, alm=T.packed(torch.cat([T.analysis(m[:1]), T.analysis2(m[1:])])))
    if kind == "pol_solve":
        return _polarised(T, q, case["tol"])
    if kind == "multi":
        return _joint(T, q["cl"], q, case["tol"])
    if kind == "iterate":
        ls, _ = inputs.alm_lm_arrays(lmax)
        start = T.dense(_alm(q["cl"], _gen(seed + 1)) * torch.from_numpy(ls <= L).to(DEV))[None]
        alm, rec = _filter(T, q["cl"], q["nv"], q["mask"], q["d"], fixed=(case["lam"], L, case["niter"]), start=start,
                           synth=synth, ana=ana)
        return dict(alm=alm, chi2=np.array([r[0] + r[1] for r in rec]), norm2=np.array([r[3] for r in rec]))
    if kind == "solve":
        alm, told = _filter(T, q["cl"], q["nv"], q["mask"], q["d"], tol=case["tol"])
        return dict(alm=alm, **told)
    if kind == "batch":
        got = [_filter(T, q["cl"], q["nv"], q["mask"], q["d"][b], tol=case["tol"], max_iter=case["max_iter"])
               for b in range(maps)]
        return dict(alm=torch.stack([a for a, _ in got]), iters=np.array([t["iters"] for _, t in got]),
                    chi2=np.array([t["chi2_prior"] + t["chi2_noise"] for _, t in got]))
    # realisations: the Wiener filter of the data; the draws come from the library's own counter-based generator
    alm, _ = _filter(T, q["cl"], q["nv"], q["mask"], q["d"], tol=case["tol"])
    return dict(cr=None, wf=alm, iters=None)
