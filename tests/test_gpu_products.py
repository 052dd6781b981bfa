"""The exact digit products of the FP64-class modes (Legendre stages, ring and
flat-column transforms) and the mixed mode's stages for batches outside the
tensor-core kernels, at the edges of their tiles and on both sides of the size
rules that choose them.

Bars: single FP64-class transforms 1e-12 (operands keep 53 bits below their
row's or column's largest value and products are summed exactly, so the error is
a few 2^-53 times the square root of the terms), the same for two routes of one
transform; 1e-10 for solves; 2e-6 for single mixed transforms."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import alm_dev, dev, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _transforms(p, alm, maps):
    B, _, nalm = alm.shape
    m_out = torch.zeros((B, 3, maps.shape[-1]), dtype=torch.float64, device="cuda")
    a_out = torch.zeros((B, 3, nalm, 2), dtype=torch.float64, device="cuda")
    p.alm2map(alm_dev(alm), m_out)
    p.map2alm(dev(maps), a_out)
    torch.cuda.synchronize()
    return m_out.cpu().numpy(), a_out.cpu().numpy().view(np.complex128)[..., 0]


# 128 ring pairs per tile (nside 64 and 65), 16 multipoles per K step, 32
# columns per tile (batches 5 and 6: 30 and 36), the smallest plans, odd nside
@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("nside,lmax,B", [(1, 2, 1), (2, 5, 6), (7, 15, 5), (17, 50, 3), (64, 127, 1), (65, 128, 2)])
def test_legendre_products(orc, nside, lmax, B, prec):
    alm, maps = W.random_alm(lmax, B, 48), W.random_maps(nside, B, 49)
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_FP64 if prec == "fp64" else dmwf.DM_FLOAT_FLOAT)
    gm, ga = _transforms(p, alm, maps)
    p.close()
    for b in (0, B - 1):
        assert rel(gm[b], orc.alm2map(nside, lmax, alm[b])) < 1e-12
        assert rel(ga[b], orc.map2alm(nside, lmax, maps[b])) < 1e-12


# Ring transforms as products against the FFT kernels (an explicit radix keeps
# them): at the rule's line, orders beyond n / 2 in the belt, odd nside, columns
# beyond one tile; then a solve, whose pass also updates the maps.
@pytest.mark.parametrize("nside,lmax,B", [(64, 128, 2), (64, 191, 3), (33, 66, 8), (91, 150, 2), (128, 383, 1)])
def test_ring_products(nside, lmax, B):
    alm, maps = W.random_alm(lmax, B, 58), W.random_maps(nside, B, 59)
    npix = 12 * nside * nside
    rng = np.random.default_rng(nside)
    cl = np.zeros((4, lmax + 1))
    cl[:3, 2:] = 1.0 / np.arange(2, lmax + 1) ** 2.0
    sigma, mask = 0.5 + rng.random((3, npix)), (rng.random(npix) > 0.2).astype(np.uint8)
    out = []
    for fft in (False, True):
        p = dmwf.Plan(nside, lmax, B)
        if fft:
            p.set_ring_radix(0)
        p.set_spectra(cl)
        p.set_noise_mask(sigma, mask)
        p.set_schedule(lambda0=100.0, n_levels=2, iters_per_level=3, check_every=2)
        s = torch.zeros((B, 3, npix), dtype=torch.float64, device="cuda")
        p.wiener_filter(dev(maps), s)
        out.append(_transforms(p, alm, maps) + (s.cpu().numpy(),))
        p.close()
    for b in range(B):
        assert rel(out[0][0][b], out[1][0][b]) < 1e-12
        assert rel(out[0][1][b], out[1][1][b]) < 1e-12
        assert rel(out[0][2][b], out[1][2][b]) < 1e-10


# Rows and columns of a flat patch as products against the FFT kernels: at the
# rule's line, batches that leave a remainder of the blocks' four, the largest grid.
@pytest.mark.parametrize("N,B", [(256, 2), (256, 5), (512, 1), (2048, 1)])
def test_flat_products(N, B):
    rng = np.random.default_rng(N + B)
    k = np.minimum(np.arange(N), N - np.arange(N)).astype(np.float64)
    S = np.zeros((4, N, N))
    S[:3] = 1.0 / (1.0 + k[:, None] ** 2 + k[None, :] ** 2)
    sigma, mask = 0.5 + rng.random((3, N * N)), (rng.random(N * N) > 0.2).astype(np.uint8)
    d = rng.standard_normal((B, 3, N * N))
    seeds = np.arange(7, 7 + B, dtype=np.uint64)
    out = []
    for fft in (False, True):
        p = dmwf.FlatPlan(N, W.FLAT_L, B)
        if fft:
            p.set_ring_radix(0)
        p.set_spectra(S)
        p.set_noise(sigma, mask, mask)
        p.set_schedule(lambda0=100.0, n_levels=2, iters_per_level=2, check_every=2)
        a = torch.zeros((B, 3, N * N // 2, 2), dtype=torch.float64, device="cuda")
        m, s, c = (torch.zeros((B, 3, N * N), dtype=torch.float64, device="cuda") for _ in range(3))
        p.map2alm(dev(d), a)
        p.alm2map(a, m)
        p.wiener_filter(dev(d), s)
        p.constrained_realization(dev(d), seeds, c)
        torch.cuda.synchronize()
        out.append([t.cpu().numpy() for t in (a, m, s, c)])
        p.close()
    for x, y, bar in zip(out[0], out[1], (1e-12, 1e-12, 1e-10, 1e-10)):
        for b in range(B):
            assert rel(x[b], y[b]) < bar


# A right-hand side that is not finite stays alone: NaN in its own results, the
# others as without it.
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_products_not_finite(bad):
    nside, lmax, B = 64, 128, 3
    alm, maps = W.random_alm(lmax, B, 68), W.random_maps(nside, B, 69)
    p = dmwf.Plan(nside, lmax, B)
    gm, ga = _transforms(p, alm, maps)
    alm[1, 0, 5] = bad
    maps[1, 2, 7000] = bad
    bm, ba = _transforms(p, alm, maps)
    p.close()
    assert np.isnan(bm[1, 0]).all() and np.isnan(ba[1, 1:]).any()
    for b in (0, 2):
        assert np.array_equal(bm[b], gm[b]) and np.array_equal(ba[b], ga[b])


# Constant maps: lambda_00 is one value on every ring, so the digits of both
# operands keep their signs and the digit sums are the largest there are: for
# the first four amplitudes (over all of them), and a sweep of one power of two.
# The monopole of c is c sqrt(4 pi); operands and values are rounded at 2^-52 of
# theirs at most, four times: bar 4e-15, a lost unit of a sum is 1e-12.
def test_products_constant_maps():
    nside, lmax, B = 256, 96, 64
    amp = np.concatenate([[0.9628561361180136, 0.8613087756796693, 0.9354665353746234, 0.6738011761632003, 2.7255],
                          0.5 * 2.0 ** np.random.default_rng(8).random(B - 5)])
    maps = np.zeros((B, 3, 12 * nside * nside))
    maps[:, 0] = amp[:, None]
    p = dmwf.Plan(nside, lmax, B)
    out = torch.zeros((B, 3, (lmax + 1) * (lmax + 2) // 2, 2), dtype=torch.float64, device="cuda")
    p.map2alm(dev(maps), out)
    torch.cuda.synchronize()
    p.close()
    mono = out[:, 0, 0, 0].cpu().numpy()
    assert np.abs(mono / (amp * np.sqrt(4.0 * np.pi)) - 1.0).max() < 4e-15


# Mixed mode outside the tensor-core batches: FP32 kernels below the size rules
# (23: ring pairs not a multiple of 4; 64, 190: the largest analysis, 100, 244:
# the largest synthesis; batch 4: four right-hand sides a thread; batch 2 above
# the line), digit products of 27 bits beyond (64, 191 and 100, 245).
@pytest.mark.parametrize("nside,lmax,B", [(1, 2, 1), (23, 60, 3), (32, 95, 4), (64, 190, 3), (64, 191, 3),
                                          (100, 244, 5), (100, 245, 5), (129, 200, 2), (128, 256, 7)])
def test_mixed_small_batches(orc, nside, lmax, B):
    alm, maps = W.random_alm(lmax, B, 78), W.random_maps(nside, B, 79)
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    gm, ga = _transforms(p, alm, maps)
    p.close()
    for b in (0, B - 1):
        assert rel(gm[b], orc.alm2map(nside, lmax, alm[b])) < 2e-6
        assert rel(ga[b], orc.map2alm(nside, lmax, maps[b])) < 2e-6


# Flat patches on both sides of the size rule of their products: at the line and
# one right-hand side below it, and a grid that never takes them.  The matrices
# show in the plan's bytes; either way the transforms agree with the FFT kernels.
@pytest.mark.parametrize("N,B,products", [(64, 70, False), (128, 63, False), (128, 64, True), (256, 3, False),
                                          (256, 4, True), (512, 1, True)])
def test_flat_size_rule(N, B, products):
    rng = np.random.default_rng(N + B)
    d = dev(rng.standard_normal((B, 3, N * N)))
    out = []
    for fft in (False, True):
        p = dmwf.FlatPlan(N, W.FLAT_L, B)
        if fft:
            p.set_ring_radix(0)
        held = p.info()["workspace_bytes"]
        a, m = torch.zeros((B, 3, N * N // 2, 2), dtype=torch.float64, device="cuda"), torch.zeros_like(d)
        p.map2alm(d, a)
        p.alm2map(a, m)
        torch.cuda.synchronize()
        assert (p.info()["workspace_bytes"] > held) == (products and not fft)
        out.append((a.cpu().numpy(), m.cpu().numpy()))
        p.close()
    for x, y in zip(*out):
        for b in (0, B - 1):
            assert rel(x[b], y[b]) < 1e-12
