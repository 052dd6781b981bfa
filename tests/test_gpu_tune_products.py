"""dm_autotune reports the ring stage that the iterations run: on an FP64-class
plan whose rings run as digit products their time (one figure, nothing to pick),
close to that of a solve's own iterations; with an explicit radix the FFT
kernels' again.  The ratio's bounds leave a factor of 1.4 to the clock and the
cache; the FFT kernels take about twice as long at this size."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("prec", [dmwf.DM_FP64, dmwf.DM_FLOAT_FLOAT])
@pytest.mark.parametrize("fft", [False, True])
def test_ring_time_is_that_of_the_iterations(prec, fft):
    nside, lmax, B = 128, 256, 8
    npix = 12 * nside * nside
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(prec)
    if fft:
        p.set_ring_radix(3)
    cl = np.zeros((4, lmax + 1))
    cl[:3, 2:] = 1.0 / np.arange(2, lmax + 1) ** 2.0
    p.set_spectra(cl)
    p.set_noise_mask(np.full((3, npix), 0.5), np.ones(npix, np.uint8))
    p.set_schedule(lambda0=10.0, n_levels=1, iters_per_level=64, check_every=32)
    d = dev(W.random_maps(nside, B, 3))
    s = torch.zeros_like(d)
    p.wiener_filter(d, s)  # its right-hand sides are finished, and count as running for the tuner all the same
    t = p.autotune(force=True)
    if not fft:
        assert t["ms_ring"] == t["ms_ring_default"]
    p.profile_enable(True)
    p.wiener_filter(d, s)
    prof = p.profile_read()
    p.close()
    run = prof["ms_ring"] / prof["iterations"]
    assert 1 / 1.4 < t["ms_ring"] / run < 1.4
