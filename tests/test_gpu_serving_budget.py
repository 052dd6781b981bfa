"""A served pool stays within the device memory that it reserves, whatever of its
budget is left for digit tables: from one that holds all of them down to the
smallest one that takes the request.  Measured as the device's free memory;
16 MiB are left to the allocator's granularity and to modules loaded meanwhile."""
import time

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _serve(budget, slots, prec, tol, wl, d):
    """(status, bytes reserved, bytes taken, map) of one request on a fresh server."""
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    srv = dmwf.Server(budget, slots_per_plan=slots, iters_per_round=16, n_levels=3, prec=dmwf.DM_MIXED_FP32,
                      strict_tol=1e-3 if prec != dmwf.DM_MIXED_FP32 else 0.0,
                      strict_prec=prec if prec != dmwf.DM_MIXED_FP32 else dmwf.DM_FP64)
    t = srv.submit(wl.nside, wl.lmax, 0, tol, wl.cl, wl.sigma, d, wl.mask, 0)
    got, t0 = None, time.time()
    while got is None and time.time() - t0 < 120:
        got = srv.poll(t)
        time.sleep(0.002)
    taken, held = free - torch.cuda.mem_get_info()[0], srv.info()["bytes_reserved"]
    srv.close()
    return got[0]["status"], held, taken, got[1]


@pytest.mark.parametrize("prec,slots,nside,lmax", [(dmwf.DM_FLOAT_FLOAT, 256, 64, 128), (dmwf.DM_FP64, 256, 64, 128),
                                                   (dmwf.DM_MIXED_FP32, 100, 64, 128), (dmwf.DM_MIXED_FP32, 3, 128, 256),
                                                   (dmwf.DM_MIXED_FP32, 8, 128, 256)])
def test_pool_within_its_reservation(orc, prec, slots, nside, lmax):
    wl = W.make_workload("nside16", [4], nside=nside, lmax=lmax)
    d = wl.data([orc.alm2map(nside, lmax, wl.alm_true[0])])[0]
    _serve(64 << 30, slots, prec, 1e-4, wl, d)  # kernels loaded
    st, most, taken, s0 = _serve(64 << 30, slots, prec, 1e-4, wl, d)
    assert st == dmwf.DM_OK and taken <= most + (16 << 20)
    budget, seen = most, 0
    while seen < 12:  # tables give way until the request no longer fits
        st, held, taken, s = _serve(budget, slots, prec, 1e-4, wl, d)
        if st != dmwf.DM_OK:
            assert st == dmwf.DM_ENOMEM
            break
        assert held <= budget + (16 << 20) and taken <= held + (16 << 20)
        assert np.linalg.norm(s - s0) < 1e-6 * np.linalg.norm(s0)
        budget, seen = int(0.96 * budget), seen + 1
    assert seen > 1
