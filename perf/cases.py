"""The work whose speed is measured: calls of the dual messenger library as its users make them.

listed() holds the configurations the framework is quoted on (the plain FP64 solve at nside 16, the
single solve at nside 256 in both arithmetic modes, the batched solves of constrained realisations at
nside 512, the paper's 1024 x 1024 flat patch, the served mix) and the calls beside them that a user
makes for their own sake (transforms, the strict float-float mode, correlated noise, odd sizes).
draw() gives more cases of the same ranges.  Spectra, noise levels, masks and the cooling schedule are
those of the repository's workloads; the signal is a Gaussian field of those spectra.

A solve runs its ten cooling levels (lambda 1000 -> 1) with a fixed count per level, so that every run
does the same iterations.  Results of the mixed mode are kept in single precision, which is what its
maps are stored in on the device; the FP64 and float-float modes return FP64.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_1801_05358_gb300 import dmwf

PREC = {"fp64": dmwf.DM_FP64, "mixed": dmwf.DM_MIXED_FP32, "ff": dmwf.DM_FLOAT_FLOAT}
LEVELS = 10
FLAT_SIDE = math.radians(10.0)


def listed():
    return [
        # the plain FP64 solve of the smallest configuration: 100 iterations, launches and latency
        dict(name="wf_fp64_nside16", op="wf", prec="fp64", nside=16, lmax=47, batch=1, iters=10),
        # one sky at nside 256, plain FP64 (what a default plan does)
        dict(name="wf_fp64_nside256", op="wf", prec="fp64", nside=256, lmax=512, batch=1, iters=2),
        # the same sky in the mixed mode, one right-hand side
        dict(name="wf_mixed_nside256", op="wf", prec="mixed", nside=256, lmax=512, batch=1, iters=20),
        # a full batch of 64 right-hand sides at the medium resolution
        dict(name="wf_mixed_nside256_b64", op="wf", prec="mixed", nside=256, lmax=512, batch=64, iters=10),
        # constrained realisations at the resolution of the headline benchmark
        dict(name="cr_mixed_nside512_b16", op="cr", prec="mixed", nside=512, lmax=1024, batch=16, iters=20),
        # a pool of the strict serving precision
        dict(name="wf_ff_nside128_b8", op="wf", prec="ff", nside=128, lmax=256, batch=8, iters=3),
        # correlated noise with distinct masks (the paper's own noise model), an odd batch
        dict(name="cov_fp64_nside64_b3", op="cov", prec="fp64", nside=64, lmax=128, batch=3, iters=3),
        # the paper's patch
        dict(name="flat_1024_b16", op="flat", prec="fp64", nside=1024, lmax=0, batch=16, iters=3),
        # a synthesis and an analysis by themselves: a large plain one, a batched mixed one above the
        # size whose Legendre tiles are stored, and a ragged geometry (nside no power of two)
        dict(name="alm2map_fp64_nside512", op="alm2map", prec="fp64", nside=512, lmax=1024, batch=1, iters=0),
        dict(name="map2alm_mixed_nside1024_b8", op="map2alm", prec="mixed", nside=1024, lmax=2048, batch=8, iters=0),
        dict(name="map2alm_fp64_nside100_b5", op="map2alm", prec="fp64", nside=100, lmax=237, batch=5, iters=0),
        # eight requests, Wiener filter and constrained realisation, to a running server
        dict(name="serve_nside64_8", op="serve", prec="mixed", nside=64, lmax=128, batch=8, iters=60),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: an operation, a precision it has, and sizes between the smallest and largest listed."""
    op = rng.choice(["wf", "wf", "cr", "cov", "flat", "alm2map", "map2alm", "map2alm", "serve"])
    if op == "flat":
        n = 2 ** rng.randint(6, 10)
        return dict(op=op, prec="fp64", nside=n, lmax=0, batch=rng.randint(1, 16), iters=rng.randint(1, 3))
    if op == "serve":
        nside = rng.choice([16, 32, 64])
        return dict(op=op, prec="mixed", nside=nside, lmax=2 * nside, batch=rng.randint(2, 8), iters=rng.randint(20, 60))
    prec = rng.choice(["fp64", "ff"] if op == "cov" else ["fp64", "mixed", "mixed", "ff"])
    nside = _log_int(rng, 16, 512 if op in ("alm2map", "map2alm") else 256)
    if rng.random() < 0.5:  # half of them powers of two, as most users' maps are
        nside = 2 ** int(math.log2(nside))
    lmax = 2 * nside if rng.random() < 0.5 else rng.randint(nside, 3 * nside - 1)
    batch = _log_int(rng, 1, 64 if nside <= 128 else (16 if nside <= 256 else 4))
    if prec != "mixed" and op not in ("alm2map", "map2alm"):  # the slow precisions solve fewer at once
        batch = max(1, batch // 4)
    iters = 0 if op in ("alm2map", "map2alm") else rng.randint(1, 3 if prec != "mixed" else 10)
    return dict(op=op, prec=prec, nside=nside, lmax=lmax, batch=batch, iters=iters)


# ----------------------------------------------------------------------------------------------
# Inputs: HEALPix geometry, spectra, noise and masks of the workloads, in torch


def _rings(nside):
    """Per ring: first pixel, pixel count, z, phi of the first pixel (RING order)."""
    i = np.arange(1, 4 * nside, dtype=np.int64)
    k = np.minimum(i, 4 * nside - i)
    cap = k < nside
    n = np.where(cap, 4 * k, 4 * nside)
    start = np.concatenate([[0], np.cumsum(n)[:-1]])
    zc = 1.0 - k.astype(np.float64) ** 2 / (3.0 * nside * nside)
    ze = 4.0 / 3.0 - 2.0 * i / (3.0 * nside)
    z = np.where(cap, np.where(i < 2 * nside, zc, -zc), ze)
    shift = np.where(cap, 0.5, 0.5 * ((i - nside + 1) % 2))
    return start, n, z, shift * 2.0 * np.pi / n


def _pixels(nside, dev):
    """z and phi of every pixel."""
    start, n, z, phi0 = _rings(nside)
    ring = torch.repeat_interleave(torch.arange(len(n), device=dev), torch.from_numpy(n).to(dev))
    j = torch.arange(12 * nside * nside, device=dev) - torch.from_numpy(start).to(dev)[ring]
    zt, nt, pt = (torch.from_numpy(np.asarray(v, dtype=np.float64)).to(dev) for v in (z, n, phi0))
    return zt[ring], pt[ring] + 2.0 * math.pi * (j / nt[ring])


def _spectra(ell, scale):
    """[4, ...] TT, EE, BB, TE at multipoles ell (the workloads' analytic spectra)."""
    pos = ell > 0
    safe = np.where(pos, ell, 1.0)
    tt = np.where(pos, np.exp(-(safe / scale) ** 2) / (safe * (safe + 1.0)), 0.0)
    ee = np.where(ell >= 2, 0.05 * tt, 0.0)
    return np.stack([tt, ee, 0.01 * ee, np.where(ell >= 2, 0.3 * np.sqrt(tt * ee), 0.0)])


def _mask(vec, z, band, gen, radii):
    obs = z.abs() >= band
    for r in radii:
        c = torch.randn(3, generator=gen, device=vec.device, dtype=torch.float64)
        obs &= (vec * (c / c.norm())[:, None]).sum(0) < math.cos(r)
    return obs


def _sphere_sky(case, gen, dev):
    """Spectra, noise, masks and data of a case; the data are signal plus noise on observed pixels."""
    nside, lmax, B = case["nside"], case["lmax"], case["batch"]
    cl = _spectra(np.arange(lmax + 1, dtype=np.float64), 40.0)
    z, phi = _pixels(nside, dev)
    sth = torch.sqrt((1.0 - z * z).clamp_min(0.0))
    vec = torch.stack([sth * torch.cos(phi), sth * torch.sin(phi), z])
    ell = np.arange(lmax + 1)
    s0 = 0.1 * math.sqrt(float(((2 * ell + 1) * cl[0]).sum()) / (4.0 * math.pi))
    u = torch.rand(z.shape, generator=gen, device=dev, dtype=torch.float64)
    st = s0 * (1.0 + 2.0 * z.abs()) * (0.5 + u)
    sigma = torch.stack([st, math.sqrt(2.0) * st, math.sqrt(2.0) * st])
    if case["op"] == "cov":
        mask = _mask(vec, z, 0.215, gen, [math.radians(3.0)] * 10)
        mask_p = _mask(vec, z, 0.175, gen, [math.radians(3.0)] * 10)
    else:
        small = [math.radians(0.5)] * 50 if nside >= 256 else []
        mask = mask_p = _mask(vec, z, 0.2, gen, [math.radians(3.0)] * 10 + small)
    rho = 0.6 * torch.rand(sigma.shape, generator=gen, device=dev, dtype=torch.float64) - 0.3
    leff = min(lmax, 160)  # the spectra are below 1e-7 of their peak beyond
    alm = _draw_alm(leff, cl, B, gen, dev)
    d = _Sphere(nside, leff, dev).synthesis(alm)
    obs = torch.stack([mask, mask_p, mask_p])
    noise = torch.randn(d.shape, generator=gen, device=dev, dtype=torch.float64)
    if case["op"] == "cov":
        noise = _correlate(noise, rho)
    d = (d + sigma * noise) * obs
    return dict(cl=cl, sigma=sigma, rho=rho, mask=mask, mask_p=mask_p, d=d.contiguous())


def _correlate(x, rho):
    """Unit normals [B, 3, npix] to the correlations (IQ, IU, QU) per pixel, by the Cholesky factor."""
    l10, l20 = rho[0], rho[1]
    l11 = torch.sqrt(1.0 - l10 * l10)
    l21 = (rho[2] - l10 * l20) / l11
    l22 = torch.sqrt(1.0 - l20 * l20 - l21 * l21)
    return torch.stack([x[:, 0], l10 * x[:, 0] + l11 * x[:, 1], l20 * x[:, 0] + l21 * x[:, 1] + l22 * x[:, 2]], 1)


def _lm(lmax):
    """l and m of every stored coefficient (m-major)."""
    ls = np.concatenate([np.arange(m, lmax + 1) for m in range(lmax + 1)])
    ms = np.concatenate([np.full(lmax + 1 - m, m) for m in range(lmax + 1)])
    return ls, ms


def _draw_alm(lmax, cl, B, gen, dev, white=False):
    """Gaussian (T, E, B) coefficients [B, 3, nalm]; white: unit spectra for every l the field has."""
    ls, ms = (torch.from_numpy(v).to(dev) for v in _lm(lmax))
    z = torch.randn((B, 3, ls.numel(), 2), generator=gen, device=dev, dtype=torch.float64)
    z[..., 1] *= (ms > 0)
    scale = torch.ones(ls.numel(), dtype=torch.float64, device=dev)
    scale[ms > 0] = math.sqrt(0.5)
    z = torch.view_as_complex(z) * scale
    if white:
        z[:, 1:] *= (ls >= 2)
        return z
    tt, ee, bb, te = (torch.from_numpy(cl[k]).to(dev)[ls] for k in range(4))
    l11 = torch.sqrt(tt)
    l21 = torch.where(l11 > 0, te / torch.where(l11 > 0, l11, 1.0), 0.0)
    l22 = torch.sqrt((ee - l21 * l21).clamp_min(0.0))
    return torch.stack([l11 * z[:, 0], l21 * z[:, 0] + l22 * z[:, 1], torch.sqrt(bb) * z[:, 2]], 1)


def _flat_sky(case, gen, dev):
    N, B = case["nside"], case["batch"]
    k = np.fft.fftfreq(N, d=1.0 / N)
    ell = 2.0 * math.pi / FLAT_SIDE * np.hypot(k[:, None], k[None, :])
    ny = (k == -(N // 2))
    S = _spectra(ell, 1500.0) * ~(ny[:, None] | ny[None, :])
    s0 = 0.04 * math.sqrt(float(S[0].sum())) / FLAT_SIDE
    st = s0 * (0.75 + 0.5 * torch.rand((N, N), generator=gen, device=dev, dtype=torch.float64))
    sigma = torch.stack([st, math.sqrt(2.0) * st, math.sqrt(2.0) * st])
    y, x = torch.meshgrid(torch.arange(N, device=dev), torch.arange(N, device=dev), indexing="ij")
    masks = []
    for count in (100, 70):  # a strip of a tenth of the patch and disks: sky fractions near 0.78 and 0.82
        m = torch.ones((N, N), dtype=torch.bool, device=dev)
        h = int(round(0.1 * N))
        m[(N - h) // 2:(N - h) // 2 + h] = False
        for c in torch.rand((count, 3), generator=gen, device=dev, dtype=torch.float64).tolist():
            r = N * (0.01 + 0.03 * c[2])
            m &= (y - c[0] * N) ** 2 + (x - c[1] * N) ** 2 >= r * r
        masks.append(m)
    z = torch.fft.fft2(torch.randn((B, 3, N, N), generator=gen, device=dev, dtype=torch.float64)) * (FLAT_SIDE / N)
    tt, ee, bb, te = (torch.from_numpy(S[i]).to(dev) for i in range(4))
    l11 = torch.sqrt(tt)
    l21 = torch.where(l11 > 0, te / torch.where(l11 > 0, l11, 1.0), 0.0)
    l22 = torch.sqrt((ee - l21 * l21).clamp_min(0.0))
    a = torch.stack([l11 * z[:, 0], l21 * z[:, 0] + l22 * z[:, 1], torch.sqrt(bb) * z[:, 2]], 1)
    d = _Flat(N, dev).synthesis(a)
    obs = torch.stack([masks[0], masks[1], masks[1]])
    d = (d + sigma * torch.randn(d.shape, generator=gen, device=dev, dtype=torch.float64)) * obs
    return dict(S=S, sigma=sigma, mask=masks[0], mask_p=masks[1], d=d.contiguous())


def _inputs(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    if case["op"] == "flat":
        return _flat_sky(case, gen, dev)
    if case["op"] == "alm2map":
        return dict(alm=_draw_alm(case["lmax"], None, case["batch"], gen, dev, white=True))
    if case["op"] == "map2alm":
        npix = 12 * case["nside"] ** 2
        return dict(map=torch.randn((case["batch"], 3, npix), generator=gen, device=dev, dtype=torch.float64))
    sky = _sphere_sky(case, gen, dev)
    sky["seeds"] = np.array([int(seed) * 1000 + b for b in range(case["batch"])], dtype=np.uint64)
    return sky


# ----------------------------------------------------------------------------------------------


def prepare(case, seed):
    """A plan set up for the case (its sky, precision and schedule), the data, and the output buffers."""
    op, B = case["op"], case["batch"]
    sky = _inputs(case, seed)
    host = lambda t: t.cpu().numpy()  # noqa: E731
    if op == "serve":
        server = dmwf.Server(hbm_budget_bytes=16 << 30, slots_per_plan=8, iters_per_round=16, prec=PREC[case["prec"]],
                             n_levels=LEVELS, max_iter=case["iters"])
        req = [dict(nside=case["nside"], lmax=case["lmax"], kind=dmwf.DM_REQ_CR if b % 3 == 2 else dmwf.DM_REQ_WF,
                    tol=1e-6, cl=sky["cl"], sigma=host(sky["sigma"]), d=host(sky["d"][b]), mask=host(sky["mask"]),
                    seed=int(sky["seeds"][b])) for b in range(B)]
        return dict(case=case, server=server, requests=req)
    if op == "flat":
        N = case["nside"]
        plan = dmwf.FlatPlan(N, FLAT_SIDE, B)
        plan.set_spectra(sky["S"])
        plan.set_noise(host(sky["sigma"]), host(sky["mask"]), host(sky["mask_p"]))
        alm_shape = (B, 3, N // 2, N)
    else:
        plan = dmwf.Plan(case["nside"], case["lmax"], B)
        alm_shape = (B, 3, plan.nalm)
        if op in ("wf", "cr"):
            plan.set_spectra(sky["cl"])
            plan.set_noise_mask(host(sky["sigma"]), host(sky["mask"]))
        elif op == "cov":
            plan.set_spectra(sky["cl"])
            plan.set_noise_cov(host(sky["sigma"]), host(sky["rho"]), host(sky["mask"]), host(sky["mask_p"]))
        plan.set_precision(PREC[case["prec"]])
    if case["iters"]:
        plan.set_schedule(lambda0=1000.0, n_levels=LEVELS, iters_per_level=case["iters"], check_every=8)
    dev = torch.device("cuda")
    state = dict(case=case, plan=plan)
    if op != "alm2map":
        state["alm"] = torch.empty(alm_shape, dtype=torch.complex128, device=dev)
    if op != "map2alm":
        state["s"] = torch.empty((B, 3, plan.npix), dtype=torch.float64, device=dev)
    state.update({k: sky[k] for k in ("d", "map", "seeds") if k in sky})
    if op == "alm2map":
        state["alm_in"] = sky["alm"]
    return state


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "serve":
        server = state["server"]
        tickets = [server.submit(**r) for r in state["requests"]]
        maps = []
        for t in tickets:
            while (done := server.poll(t)) is None:
                time.sleep(0.0002)
            maps.append(done[1].astype(np.float32))
        return maps
    plan = state["plan"]
    if op == "alm2map":
        plan.alm2map(state["alm_in"], state["s"])
        out = [state["s"]]
    elif op == "map2alm":
        plan.map2alm(state["map"], state["alm"])
        out = [state["alm"]]
    elif op == "cr":
        plan.constrained_realization(state["d"], state["seeds"], state["s"], state["alm"])
        out = [state["s"], state["alm"]]
    else:
        plan.wiener_filter(state["d"], state["s"], state["alm"])
        out = [state["s"], state["alm"]]
    if case["prec"] == "mixed":
        out = [x.to(torch.complex64 if x.is_complex() else torch.float32) for x in out]
    return out


def work(case):
    """Inputs read and outputs written once; the transforms' operations (20 per l, m, ring pair and
    right-hand side for each Legendre stage, 2.5 n log2 n for a real transform of n points)."""
    op, B = case["op"], case["batch"]
    iters = LEVELS * case["iters"] if op != "serve" else case["iters"]
    if op == "flat":
        N = case["nside"]
        maps, alms = 3.0 * N * N * 8, 3.0 * (N // 2) * N * 16
        fft = 3 * 2.5 * N * N * 2 * math.log2(N)
        leg = 0.0
    else:
        nside, lmax = case["nside"], case["lmax"]
        npix, nalm = 12.0 * nside * nside, (lmax + 1) * (lmax + 2) / 2.0
        maps, alms = 3 * npix * 8, 3 * nalm * 16
        fft = 3 * sum(2.5 * n * math.log2(n) for n in _rings(nside)[1].tolist())
        leg = 20.0 * nalm * 2 * nside
    if op in ("alm2map", "map2alm"):
        return {"bytes": B * (maps + alms), "flops": B * (leg + fft)}
    passes = 2.0 * iters
    # d and s, sigma and the harmonic coefficients; the schedule's transforms
    return {"bytes": B * (2 * maps + (alms if op != "serve" else 0)) + maps, "flops": passes * B * (leg + fft)}


# ----------------------------------------------------------------------------------------------
# The same in 64 bits with torch alone


class _Sphere:
    """Spin-0 and spin-2 transforms of a HEALPix grid: Wigner-d recurrences in l over every (m, ring
    pair), one batched product per l, and one FFT per ring length.  (Q +- iU) = sum -(aE +- i aB) +-2Y."""

    def __init__(self, nside, lmax, dev):
        self.nside, self.lmax, self.dev = nside, lmax, dev
        start, n, z, phi0 = _rings(nside)
        self.start, self.n, self.phi0 = start, n, phi0
        self.npairs = 2 * nside
        i = np.arange(1, 2 * nside + 1)
        th = np.where(i < nside, 2.0 * np.arcsin(i / (nside * math.sqrt(6.0))), np.arccos(z[:2 * nside]))
        self.th = torch.from_numpy(th).to(dev)
        m = np.arange(lmax + 1)
        self.base = torch.from_numpy(m * (2 * lmax + 1 - m) // 2).to(dev)
        self.kept = None

    def _seeds(self, k):
        """d^l0_{m,k} at l0 = max(m, |k|) for every m, [lmax + 1, npairs]."""
        m = torch.arange(self.lmax + 1, device=self.dev, dtype=torch.float64)[:, None]
        s, c = torch.sin(self.th / 2)[None], torch.cos(self.th / 2)[None]
        if k == 0:
            ratio = torch.where(m > 0, torch.sqrt((2 * m - 1).clamp_min(0) / (2 * m).clamp_min(1)), 1.0)
            out = torch.cumprod(torch.where(m > 0, -2 * s * c, torch.ones_like(s)) * ratio, 0)
            return out
        mm = m.clamp_min(3)  # d^m from d^{m-1}: sqrt(2m (2m - 1) / ((m + k)(m - k))) sin cos
        step = torch.where(m >= 3, -torch.sqrt(2 * mm * (2 * mm - 1) / ((mm + k) * (mm - k))) * s * c, torch.ones_like(s * c))
        step[2] = (c if k > 0 else s) ** 4
        out = torch.ones_like(step)
        out[2:] = torch.cumprod(step[2:], 0)
        out[0] = math.sqrt(6.0) * (s * c) ** 2
        out[1] = (2 * s * c ** 3) if k > 0 else (-2 * s ** 3 * c)
        return out

    def keep(self):
        """Hold the values of every l for the transforms that follow."""
        self.kept = [tuple(v.clone() if k else v for k, v in enumerate(x)) for x in self._values()]
        return self

    def _values(self):
        """For l = 0 .. lmax: (l, lambda, 2lambda, -2lambda), each [l + 1, npairs]."""
        if self.kept is not None:
            yield from self.kept
            return
        L, dev = self.lmax, self.dev
        x = torch.cos(self.th)[None]
        mf = torch.arange(L + 1, device=dev, dtype=torch.float64)[:, None]
        seeds = [self._seeds(k) for k in (0, -2, 2)]
        cur = [torch.zeros_like(seeds[0]) for _ in range(3)]
        prev = [torch.zeros_like(seeds[0]) for _ in range(3)]
        for l in range(L + 1):
            if l > 0:
                j = l - 1.0  # from j to l
                for f, k in enumerate((0, -2, 2)):
                    if k != 0 and l <= 2:
                        continue
                    m = mf[:l]
                    den = torch.sqrt((l * l - m * m) * (l * l - k * k))
                    if k == 0:
                        new = ((2 * j + 1) * x * cur[f][:l] - torch.sqrt((j * j - m * m).clamp_min(0)) * prev[f][:l]) / torch.sqrt(l * l - m * m)
                    else:
                        new = ((2 * j + 1) * (j * l * x - m * k) * cur[f][:l]
                               - l * torch.sqrt((j * j - m * m).clamp_min(0) * (j * j - k * k)) * prev[f][:l]) / (j * den)
                    prev[f][:l] = cur[f][:l]
                    cur[f][:l] = new
            for f, k in enumerate((0, -2, 2)):
                if k == 0 or l > 2:
                    cur[f][l] = seeds[f][l]
                elif l == 2:
                    cur[f][:3] = seeds[f][:3]
            nl = math.sqrt((2 * l + 1) / (4 * math.pi))
            yield (l,) + tuple(nl * cur[f][:l + 1] for f in range(3))

    def _groups(self):
        """Ring numbers by length: (n, rings, phi0)."""
        by = {}
        for r, n in enumerate(self.n.tolist()):
            by.setdefault((n, round(self.phi0[r] * n, 6)), []).append(r)
        return [(key[0], rs, float(self.phi0[rs[0]])) for key, rs in by.items()]

    def synthesis(self, alm):
        """[B, 3, nalm] -> [B, 3, npix]"""
        B, L, P, ns = alm.shape[0], self.lmax, self.npairs, self.nside
        F = torch.zeros((6, B, L + 1, P), dtype=torch.complex128, device=self.dev)  # T, +, - of north, then south
        for l, t, p, q in self._values():
            idx = self.base[:l + 1] + l
            a = alm[:, :, idx]
            ap, am = -(a[:, 1] + 1j * a[:, 2]), -(a[:, 1] - 1j * a[:, 2])
            sg = 1.0 - 2.0 * ((torch.arange(l + 1, device=self.dev) + l) % 2)
            for o, (v, c) in enumerate(((t, a[:, 0]), (p, ap), (q, am))):
                F[o, :, :l + 1] += c[..., None] * v
            for o, (v, c) in enumerate(((t, a[:, 0]), (q, ap), (p, am))):
                F[3 + o, :, :l + 1] += (c * sg)[..., None] * v
        out = torch.empty((B, 3, 12 * ns * ns), dtype=torch.float64, device=self.dev)
        m = torch.arange(L + 1, device=self.dev)
        for n, rs, phi0 in self._groups():
            e = torch.exp(1j * phi0 * m.double())
            for side in (0, 1):
                rings = [r for r in rs if (r < P) == (side == 0)]
                if not rings:
                    continue
                pr = [r if r < P else 4 * ns - 2 - r for r in rings]
                G = F[3 * side:3 * side + 3, :, :, pr]
                g = torch.stack([G[0], (G[1] + G[2]) / 2, (G[1] - G[2]) / 2j], 1)  # [B, 3, m, ring]
                g = (g * e[:, None]).transpose(2, 3)
                H = torch.zeros(g.shape[:3] + (n,), dtype=torch.complex128, device=self.dev)
                H.index_add_(3, m % n, g)
                H.index_add_(3, (-m[1:]) % n, g[..., 1:].conj())
                v = torch.fft.ifft(H, dim=3).real * n
                for j, r in enumerate(rings):
                    out[:, :, self.start[r]:self.start[r] + n] = v[:, :, j]
        return out

    def analysis(self, maps):
        """Omega Y^dagger: [B, 3, npix] -> [B, 3, nalm]"""
        B, L, P, ns = maps.shape[0], self.lmax, self.npairs, self.nside
        G = torch.zeros((6, B, L + 1, P), dtype=torch.complex128, device=self.dev)
        m = torch.arange(L + 1, device=self.dev)
        for n, rs, phi0 in self._groups():
            e = torch.exp(-1j * phi0 * m.double())
            v = torch.stack([maps[:, :, self.start[r]:self.start[r] + n] for r in rs], 2)
            h = torch.fft.fft(v.to(torch.complex128), dim=3)[..., m % n] * e  # [B, 3, ring, m]
            for side in (0, 1):
                at = [j for j, r in enumerate(rs) if (r < P) == (side == 0)]
                if not at:
                    continue
                pr = [rs[j] if side == 0 else 4 * ns - 2 - rs[j] for j in at]
                g = h[:, :, at].transpose(2, 3)
                G[3 * side, :, :, pr] = g[:, 0]
                G[3 * side + 1, :, :, pr] = g[:, 1] + 1j * g[:, 2]
                G[3 * side + 2, :, :, pr] = g[:, 1] - 1j * g[:, 2]
        alm = torch.zeros((B, 3, (L + 1) * (L + 2) // 2), dtype=torch.complex128, device=self.dev)
        om = 4.0 * math.pi / (12.0 * ns * ns)
        for l, t, p, q in self._values():
            idx = self.base[:l + 1] + l
            sg = 1.0 - 2.0 * ((torch.arange(l + 1, device=self.dev) + l) % 2)
            N, S = G[:3, :, :l + 1], G[3:, :, :l + 1]
            alm[:, 0, idx] = om * ((N[0] * t).sum(-1) + sg * (S[0] * t).sum(-1))
            gp = (N[1] * p).sum(-1) + sg * (S[1] * q).sum(-1)
            gm = (N[2] * q).sum(-1) + sg * (S[2] * p).sum(-1)
            alm[:, 1, idx] = -om * (gp + gm) / 2
            alm[:, 2, idx] = -om * (gp - gm) / 2j
        return alm


class _Flat:
    """The flat patch's pair: 2-D FFT and the E/B rotation, the Nyquist row and column left out."""

    def __init__(self, N, dev):
        self.N = N
        k = torch.fft.fftfreq(N, d=1.0 / N, device=dev, dtype=torch.float64)
        ky, kx = torch.meshgrid(k, k, indexing="ij")
        phi = torch.atan2(ky, kx)
        self.c, self.s = torch.cos(2 * phi), torch.sin(2 * phi)
        self.keep = (kx != -(N // 2)) & (ky != -(N // 2))

    def analysis(self, maps):
        h = (FLAT_SIDE / self.N) ** 2 * torch.fft.fft2(maps) * self.keep
        return torch.stack([h[:, 0], h[:, 1] * self.c + h[:, 2] * self.s, -h[:, 1] * self.s + h[:, 2] * self.c], 1)

    def synthesis(self, a):
        a = a * self.keep
        h = torch.stack([a[:, 0], a[:, 1] * self.c - a[:, 2] * self.s, a[:, 1] * self.s + a[:, 2] * self.c], 1)
        return torch.fft.ifft2(h).real * (self.N / FLAT_SIDE) ** 2


def _filters(cl, mu, th):
    """(f_TT, f_TE, f_EE, f_BB): max(S_e, mu) / (max(S_e, mu) + T_h) on the eigenvalues of each block."""
    tt, ee, bb, te = cl
    mean, diff = (tt + ee) / 2, (tt - ee) / 2
    root = torch.sqrt(diff * diff + te * te)
    ang = 0.5 * torch.atan2(te, diff)  # the eigenvectors (cos, sin) and (-sin, cos)
    c, s = torch.cos(ang), torch.sin(ang)
    f1, f2, fb = (x / (x + th) for x in (v.clamp_min(max(mu, 0.0)) for v in (mean + root, mean - root, bb)))
    return f1 * c * c + f2 * s * s, (f1 - f2) * c * s, f1 * s * s + f2 * c * c, fb


def _solve(case, sky, pair, cl, omega):
    """Algorithm 1 with the fixed counts of the case: a <- F [a + A (t - s)], s = Y a."""
    d = sky["d"]
    obs = torch.stack([sky["mask"], sky["mask_p"], sky["mask_p"]])
    if case["op"] == "cov":
        rho, sg = sky["rho"], sky["sigma"]
        C = torch.ones(rho.shape[1:] + (3, 3), dtype=torch.float64, device=d.device)
        for k, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
            C[:, i, j] = C[:, j, i] = rho[k]
        inv = (obs / sg).T
        ninv = inv[:, :, None] * torch.linalg.inv(C) * inv[:, None, :]
        q = ninv.diagonal(dim1=1, dim2=2).mean(1)  # the largest eigenvalue of each 3 x 3 block, trigonometric form
        D = ninv - q[:, None, None] * torch.eye(3, dtype=torch.float64, device=d.device)
        p = torch.sqrt((D * D).sum((1, 2)) / 6.0)
        det = (D[:, 0] * torch.linalg.cross(D[:, 1], D[:, 2])).sum(1) / (2.0 * torch.where(p > 0, p, 1.0) ** 3)
        alpha = 1.0 / float((q + 2.0 * p * torch.cos(torch.acos(det.clamp(-1.0, 1.0)) / 3.0)).max())
        update = lambda x: torch.einsum("pij,bjp->bip", alpha * ninv, x)  # noqa: E731
    else:
        var = sky["sigma"] ** 2
        alpha = float(var[obs].min())
        w = torch.where(obs, alpha / var, 0.0)
        update = lambda x: w * x  # noqa: E731
    th = alpha * omega
    r, a, s = d * obs, 0.0, None
    for k in range(LEVELS):
        lam = 1.0 if k == LEVELS - 1 else 1000.0 ** (1.0 - k / (LEVELS - 1))
        f = _filters(cl, (lam - 1.0) * th, th)
        for _ in range(case["iters"]):
            t = a + pair.analysis(r)
            a = torch.stack([f[0] * t[:, 0] + f[1] * t[:, 1], f[1] * t[:, 0] + f[2] * t[:, 1], f[3] * t[:, 2]], 1)
            s = pair.synthesis(a)
            r = update(d - s)
    return s, a


def exact(case, seed):
    op, dev = case["op"], torch.device("cuda")
    if op in ("cr", "serve"):
        return None  # their draws come from the library's own generator
    if op == "flat":
        sky = _inputs(case, seed)
        N = case["nside"]
        cl = [torch.from_numpy(v).to(dev) for v in sky["S"]]
        s, a = _solve(case, sky, _Flat(N, dev), cl, (FLAT_SIDE / N) ** 2)
        a = a.transpose(2, 3)[:, :, :N // 2]  # kx < N/2 major, every ky
        return [s.reshape(s.shape[0], 3, -1), a.contiguous()]
    transforms = 1 if op in ("alm2map", "map2alm") else 2 * LEVELS * case["iters"]
    cost = transforms * (case["lmax"] * 2e-4 + case["nside"] * 5e-4)  # the loops over l and over ring lengths
    cost += transforms * case["batch"] * 1.5e-9 * case["lmax"] ** 2 * case["nside"]
    if cost > 15.0 or case["batch"] * case["lmax"] * case["nside"] > 1 << 24:
        return None
    sky = _inputs(case, seed)
    pair = _Sphere(case["nside"], case["lmax"], dev)
    if op == "alm2map":
        return [pair.synthesis(sky["alm"])]
    if op == "map2alm":
        return [pair.analysis(sky["map"])]
    pair = pair.keep()
    ls = torch.from_numpy(_lm(case["lmax"])[0]).to(dev)
    cl = [torch.from_numpy(v).to(dev)[ls] for v in sky["cl"]]
    return list(_solve(case, sky, pair, cl, 4.0 * math.pi / (12.0 * case["nside"] ** 2)))
