"""Right-hand sides that are finished cost the ring products of a batch nothing,
and those that go on are not disturbed by them: iterations after the last one of
a solve against its own (profiled ring time), and a batch whose members stop at
different iterations against the FFT kernels (1e-10, the bar of FP64 solves)."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import dev, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _plan(nside, lmax, B):
    p = dmwf.Plan(nside, lmax, B)
    cl = np.zeros((4, lmax + 1))
    cl[:3, 2:] = 1.0 / np.arange(2, lmax + 1) ** 2.0
    p.set_spectra(cl)
    npix = 12 * nside * nside
    p.set_noise_mask(np.full((3, npix), 0.5), np.ones(npix, np.uint8))
    return p


# Four launched iterations follow each of these solves' own (the polls come
# later): r of a running and e of a finished iteration from 1 r + 4 e and
# 9 r + 4 e.  Finished, the launches remain: a quarter is far above them.
def test_iterations_after_the_end():
    nside, B = 128, 8
    p = _plan(nside, 256, B)
    d = dev(W.random_maps(nside, B, 3))
    s = torch.zeros_like(d)
    ms = []
    for n in (9, 1, 9):  # the first makes the tables
        p.set_schedule(lambda0=10.0, n_levels=1, iters_per_level=n, check_every=64)
        p.wiener_filter(d, s)
        p.profile_enable(True)
        p.wiener_filter(d, s)
        ms.append(p.profile_read()["ms_ring"])
        p.profile_enable(False)
    p.close()
    r = (ms[2] - ms[1]) / 8
    assert (ms[1] - r) / 4 < 0.25 * r


@pytest.mark.parametrize("nside,lmax,B", [(64, 128, 8), (33, 70, 19)])
def test_members_that_stop_apart(nside, lmax, B):
    npix = 12 * nside * nside
    rng = np.random.default_rng(5)
    masks = [(rng.random(npix) > 0.9 * b / B).astype(np.uint8) for b in range(B)]
    d = dev(W.random_maps(nside, B, 9))
    out = []
    for fft in (False, True):
        p = _plan(nside, lmax, B)
        if fft:
            p.set_ring_radix(0)
        for b in range(B):
            p.set_noise_mask_rhs(b, np.full((3, npix), 0.3 + 0.2 * b), masks[b])
        p.set_schedule(lambda0=10.0, n_levels=2, iters_per_level=0, eps0=1e-2, eps_final=1e-4, check_every=3)
        s = torch.zeros_like(d)
        _, stats = p.wiener_filter(d, s)
        out.append((s.cpu().numpy(), [x["iters_total"] for x in stats]))
        p.close()
    assert out[0][1] == out[1][1] and len(set(out[0][1])) > 1
    for b in range(B):
        assert rel(out[0][0][b], out[1][0][b]) < 1e-10
