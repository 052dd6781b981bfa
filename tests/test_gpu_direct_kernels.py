"""The FP64 kernels that run where no digit tables can be made (no memory, first
use inside a stream capture): both Legendre stages, the FFT ring stages, the
analysis with fewer partial-sum slots than pair chunks (the chunks then run in
waves, slot 0 keeping the running sum), solves of every mode whose FP64-class
part runs through them, and captured calls.  Tables find no memory here
(dm_test_table_memory), so that none of the tensor-core products can run.  Bars:
1e-12 for FP64-class transforms, 1e-10 and 1e-5 for FP64-class and mixed solves."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import alm_dev, dev, make_plan, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# 4 and 8 chunks of 64 ring pairs, in waves of 2 and 3 slots and at once
@pytest.mark.parametrize("prec", [dmwf.DM_FP64, dmwf.DM_FLOAT_FLOAT])
@pytest.mark.parametrize("nside,slots", [(128, 2), (128, 3), (128, 8), (256, 2), (256, 3)])
def test_transforms(orc, nside, slots, prec):
    lmax, B = 2 * nside, 2
    alm, maps = W.random_alm(lmax, B, 70), W.random_maps(nside, B, 71)
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(prec)
    p.test_table_memory(0)
    p.set_analysis_slots(slots)
    held = p.info()["workspace_bytes"]
    m = torch.zeros((B, 3, 12 * nside * nside), dtype=torch.float64, device="cuda")
    a = torch.zeros((B, 3, alm.shape[-1], 2), dtype=torch.float64, device="cuda")
    p.alm2map(alm_dev(alm), m)
    p.map2alm(dev(maps), a)
    torch.cuda.synchronize()
    assert p.info()["workspace_bytes"] == held  # nothing was made: the direct kernels ran
    ga = a.cpu().numpy().view(np.complex128)[..., 0]
    p.close()
    for b in range(B):
        assert rel(m[b].cpu().numpy(), orc.alm2map(nside, lmax, alm[b])) < 1e-12
        assert rel(ga[b], orc.map2alm(nside, lmax, maps[b])) < 1e-12


@pytest.mark.parametrize("prec,B,bar", [(dmwf.DM_FP64, 2, 1e-10), (dmwf.DM_FLOAT_FLOAT, 2, 1e-10),
                                        (dmwf.DM_MIXED_FP32, 8, 1e-5)])
def test_solves_in_waves(orc, prec, B, bar):
    wl = W.make_workload("nside16", list(range(7, 7 + B)), nside=128, lmax=256)
    d = np.stack([wl.data([orc.alm2map(wl.nside, wl.lmax, a)])[0] for a in wl.alm_true])
    lam = W.lambda_schedule(1000.0, 2)
    p = make_plan(wl, B, lambda0=1000.0, n_levels=2, iters_per_level=2, check_every=8)
    p.set_precision(prec)
    p.set_refinement(2)
    p.test_table_memory(0)
    p.set_analysis_slots(3)
    s = torch.zeros((B, 3, wl.npix), dtype=torch.float64, device="cuda")
    p.wiener_filter(dev(d), s)
    p.close()
    for b in (0, B - 1):
        ref = orc.dm_solve(wl.nside, wl.lmax, wl.cl, wl.sigma, wl.mask, d[b], lam, forced_iters=[2, 2])
        assert rel(s[b].cpu().numpy(), ref["s"]) < bar


# The first call of a plan inside a capture: the direct kernels are recorded, and
# a replay after the tables have been made gives the same bits as before.
@pytest.mark.parametrize("forward", [False, True])
def test_first_call_captured(orc, forward):
    nside, lmax, B = 64, 128, 2
    alm, maps = W.random_alm(lmax, B, 72), W.random_maps(nside, B, 73)
    da, dm = alm_dev(alm), dev(maps)
    p = dmwf.Plan(nside, lmax, B)
    out = torch.zeros((B, 3, alm.shape[-1], 2) if forward else (B, 3, maps.shape[-1]), dtype=torch.float64, device="cuda")
    call = (lambda: p.map2alm(dm, out)) if forward else (lambda: p.alm2map(da, out))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    g.replay()
    first = out.clone()
    call()  # outside: the tables are made
    products = out.clone()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, first)
    for got in (first, products):
        x = got.cpu().numpy().view(np.complex128)[..., 0] if forward else got.cpu().numpy()
        for b in range(B):
            ref = orc.map2alm(nside, lmax, maps[b]) if forward else orc.alm2map(nside, lmax, alm[b])
            assert rel(x[b], ref) < 1e-12
    del g
    p.close()
