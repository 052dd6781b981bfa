"""A served result does not depend on what its pool has served before, whatever
memory the pool has for tables: the first request of a fresh server against the
same request after another one, bit for bit, at budgets from one that holds every
table down to the smallest one that takes the request."""
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


def _one(srv, wl, d):
    t = srv.submit(wl.nside, wl.lmax, 0, 1e-4, wl.cl, wl.sigma, d, wl.mask, 0)
    got, t0 = None, time.time()
    while got is None and time.time() - t0 < 120:
        got = srv.poll(t)
        time.sleep(0.001)
    return got[0]["status"], got[0]["iters"], got[1], srv.info()["bytes_reserved"]


@pytest.mark.parametrize("strict,nside,lmax,slots,step", [(dmwf.DM_FLOAT_FLOAT, 4, 8, 4, 0.0005), (dmwf.DM_FP64, 4, 8, 4, 0.0005),
                                                          (None, 16, 32, 3, 0.002), (None, 64, 128, 8, 0.02)])
def test_first_and_later_requests(orc, strict, nside, lmax, slots, step):
    wl = W.make_workload("nside16", [4, 5], nside=nside, lmax=lmax)
    d = [wl.data([orc.alm2map(nside, lmax, a)])[0] for a in wl.alm_true]
    kw = dict(slots_per_plan=slots, iters_per_round=16, n_levels=3, prec=dmwf.DM_MIXED_FP32)
    if strict is not None:
        kw.update(strict_tol=1e-3, strict_prec=strict)
    budget, seen = 16 << 30, 0
    while seen < 24:
        with dmwf.Server(budget, **kw) as srv:
            status, *first, held = _one(srv, wl, d[1])
        if status != dmwf.DM_OK:
            assert status == dmwf.DM_ENOMEM
            break
        with dmwf.Server(budget, **kw) as srv:
            _one(srv, wl, d[0])
            status, *later, _ = _one(srv, wl, d[1])
        assert status == dmwf.DM_OK and first[0] == later[0] and np.array_equal(first[1], later[1])
        budget, seen = int(min(budget, held) * (1 - step)), seen + 1
    assert seen > 1
