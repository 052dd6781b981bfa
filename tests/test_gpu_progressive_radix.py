"""An explicit ring radix holds on the plans of a progressive solve's working
resolutions too: they then run the FFT kernels and make no DFT matrices (seen in
the device's memory beyond what the main plan reports), also when the call comes
after a solve has made them."""
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


def _level_bytes(radix, later):
    """Device bytes that a progressive solve adds beyond the main plan's own."""
    nside, lmax, B = 128, 256, 8
    npix = 12 * nside * nside
    p = dmwf.Plan(nside, lmax, B)
    cl = np.zeros((4, lmax + 1))
    cl[:3, 2:] = 1.0 / np.arange(2, lmax + 1) ** 2.0
    p.set_spectra(cl)
    p.set_noise_mask(np.full((3, npix), 0.5), np.ones(npix, np.uint8))
    p.set_schedule(lambda0=1000.0, n_levels=2, iters_per_level=1, check_every=1)
    p.set_progressive(0.25, 120)
    d = dev(W.random_maps(nside, B, 3))
    s = torch.zeros_like(d)
    if radix is not None and not later:
        p.set_ring_radix(radix)
    torch.cuda.synchronize()
    free, own = torch.cuda.mem_get_info()[0], p.info()["workspace_bytes"]
    p.wiener_filter(d, s)
    if later:
        p.set_ring_radix(radix)
        p.wiener_filter(d, s)
    torch.cuda.synchronize()
    assert p.progressive_levels(2)[0][0] < nside
    added = (free - torch.cuda.mem_get_info()[0]) - (p.info()["workspace_bytes"] - own)
    p.close()
    return added


def test_radix_reaches_the_level_plans():
    _level_bytes(None, False)  # allocations of the first solve in a process
    products = _level_bytes(None, False)
    for later in (False, True):
        assert products - _level_bytes(3, later) > 16 << 20
