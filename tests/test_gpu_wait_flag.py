"""A bounded wait of a tensor-core kernel that gave up reaches the caller,
wherever in a call it happened: the flag such a kernel sets is set by the host
here.  The solve calls report it after their last synthesis and diagnostics, a
served request ends with it, and the next call or request is normal."""
import time

import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import dev, make_plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("prec", [dmwf.DM_FP64, dmwf.DM_MIXED_FP32, dmwf.DM_FLOAT_FLOAT])
def test_end_of_a_solve(orc, prec):
    wl = W.make_workload("nside16", [3])
    d = dev(wl.data([orc.alm2map(wl.nside, wl.lmax, wl.alm_true[0])]))
    p = make_plan(wl, 1, lambda0=100.0, n_levels=2, iters_per_level=2)
    p.set_precision(prec)
    s, t = torch.zeros_like(d), torch.zeros_like(d)
    p.test_wait_flag()  # of an earlier call: does not count
    p.wiener_filter(d, s)
    p.solve_begin(d)
    p.solve_iterate(100)
    p.test_wait_flag()  # as if the last synthesis had given up
    with pytest.raises(dmwf.DmError) as ei:
        p.solve_end(t)
    assert ei.value.status == dmwf.DM_ETIMEOUT
    p.wiener_filter(d, t)
    assert torch.equal(s, t)
    p.close()


def _wait(srv, tickets):
    out, t0 = {}, time.time()
    while len(out) < len(tickets) and time.time() - t0 < 120:
        for t in tickets:
            if t not in out:
                got = srv.poll(t)
                if got is not None:
                    out[t] = got
        time.sleep(0.002)
    assert len(out) == len(tickets)
    return [out[t] for t in tickets]


@pytest.mark.parametrize("prec", [dmwf.DM_FP64, dmwf.DM_MIXED_FP32])
@pytest.mark.parametrize("where", [1, 2])
def test_served_requests(orc, prec, where):
    wl = W.make_workload("nside16", [4])
    d = wl.data([orc.alm2map(wl.nside, wl.lmax, wl.alm_true[0])])[0]
    srv = dmwf.Server(8 << 30, slots_per_plan=2, iters_per_round=16, prec=prec)

    def submit():
        return srv.submit(wl.nside, wl.lmax, 0, 1e-4, wl.cl, wl.sigma, d, wl.mask, 0)

    (r0, s0), = _wait(srv, [submit()])
    assert r0["status"] == dmwf.DM_OK
    assert srv.test_wait_flag(where) == dmwf.DM_OK
    (r1, _), = _wait(srv, [submit()])
    assert r1["status"] == dmwf.DM_ETIMEOUT
    (r2, s2), = _wait(srv, [submit()])
    assert r2["status"] == dmwf.DM_OK and np.array_equal(s2, s0)
    srv.close()
