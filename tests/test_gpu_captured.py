"""Stage calls recorded into CUDA graphs: whatever the plan runs afterwards (a
solve, whose anchors need more scratch than the recorded call; other tensor-core
tiles), a replay finds the memory that the recorded launches name, and gives the
plain call's result bit for bit (the same launches on the same inputs)."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import alm_dev, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _captured(call):
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


# Three digits recorded, six needed by the solve's anchors (batch 3), and both
# directions; the scratch is made once, so the plan's bytes stay where they were.
@pytest.mark.parametrize("forward", [False, True])
def test_replay_after_a_solve(forward):
    nside, lmax, B = 128, 256, 3
    npix, nalm = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    p.set_ring_radix(3)  # FFT anchors: no ring tables are added by the solve
    p.set_diagnostics(False)
    cl = np.zeros((4, lmax + 1))
    cl[:3, 2:] = 1.0 / np.arange(2, lmax + 1) ** 2.0
    p.set_spectra(cl)
    p.set_noise_mask(np.full((3, npix), 0.5), np.ones(npix, np.uint8))
    p.set_schedule(lambda0=10.0, n_levels=2, iters_per_level=2, check_every=2)
    alm, maps = alm_dev(W.random_alm(lmax, B, 5)), dev(W.random_maps(nside, B, 6))
    out = torch.zeros((B, 3, nalm, 2) if forward else (B, 3, npix), dtype=torch.float64, device="cuda")
    call = (lambda: p.map2alm(maps, out)) if forward else (lambda: p.alm2map(alm, out))
    g = _captured(call)
    want, held = out.clone(), p.info()["workspace_bytes"]
    p.wiener_filter(maps, torch.zeros_like(maps))
    assert p.info()["workspace_bytes"] == held
    out.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    del g
    p.close()


# Stored tiles recorded, then generated ones made (their own list of first K steps).
def test_replay_after_other_tiles():
    nside, lmax, B = 64, 128, 8
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    p.set_tc_tiles(0)
    maps = dev(W.random_maps(nside, B, 7))
    out = torch.zeros((B, 3, (lmax + 1) * (lmax + 2) // 2, 2), dtype=torch.float64, device="cuda")
    g = _captured(lambda: p.map2alm(maps, out))
    want = out.clone()
    p.set_tc_tiles(1)
    p.map2alm(maps, torch.zeros_like(out))
    out.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    del g
    p.close()
