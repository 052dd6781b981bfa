"""The calls that return coefficients keep every value's own precision: ring
coefficients of a red spectrum near the poles, and multipoles of ring
coefficients that live near the poles, many orders below the largest of their
order.  Value by value against the oracle's FP64 recurrence: all terms of these
sums have one sign, so each is good to some 1e-13 (the recurrence's growth over
64 multipoles); bar 1e-11, in the mixed mode (24 bits each) 1e-4."""
import numpy as np
import pytest

from tests.gpu_helpers import alm_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402

NSIDE, LMAX = 32, 64


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _alm_index():
    l = np.concatenate([np.arange(m, LMAX + 1) for m in range(LMAX + 1)])
    m = np.concatenate([np.full(LMAX + 1 - k, k) for k in range(LMAX + 1)])
    return l, m


def _worst(got, ref, floor):
    keep = np.abs(ref) > floor
    assert keep.any()
    return (np.abs(got - ref)[keep] / np.abs(ref)[keep]).max()


@pytest.mark.parametrize("prec,bar,floor", [(dmwf.DM_FP64, 1e-11, 1e-200), (dmwf.DM_FLOAT_FLOAT, 1e-11, 1e-200),
                                            (dmwf.DM_MIXED_FP32, 1e-4, 1e-24)])
@pytest.mark.parametrize("B", [1, 2])
def test_synthesis_near_the_poles(orc, prec, bar, floor, B):
    l, m = _alm_index()
    alm = np.zeros((B, 3, l.size), complex)
    alm[:, 0] = np.exp(-(l / 8.0) ** 2)
    alm[:, 1] = np.where(l >= 2, alm[:, 0], 0.0)
    p = dmwf.Plan(NSIDE, LMAX, B)
    p.set_precision(prec)
    rc = torch.zeros((B, 3, 4 * NSIDE - 1, LMAX + 1, 2), dtype=torch.float64, device="cuda")
    p.legendre_synthesis(alm_dev(alm), rc)
    got = rc.cpu().numpy().view(np.complex128)[..., 0]
    p.close()
    ref = orc.legendre_synthesis(NSIDE, LMAX, alm[0])
    for b in range(B):  # the first rings, orders well above l sin(theta)
        assert _worst(got[b][:, :4, 10:], ref[:, :4, 10:], floor) < bar


# lambda_lm of the lowest multipoles of an order, at the polar rings alone
@pytest.mark.parametrize("prec,bar,floor", [(dmwf.DM_FP64, 1e-11, 1e-200), (dmwf.DM_FLOAT_FLOAT, 1e-11, 1e-200),
                                            (dmwf.DM_MIXED_FP32, 1e-4, 1e-24)])
def test_analysis_of_polar_rings(orc, prec, bar, floor):
    l, m = _alm_index()
    rc = np.zeros((2, 3, 4 * NSIDE - 1, LMAX + 1), complex)
    rc[:, 0, :4] = 1.0
    p = dmwf.Plan(NSIDE, LMAX, 2)
    p.set_precision(prec)
    out = torch.zeros((2, 3, l.size, 2), dtype=torch.float64, device="cuda")
    p.legendre_analysis(alm_dev(rc), out)
    got = out.cpu().numpy().view(np.complex128)[..., 0]
    p.close()
    ref = orc.legendre_analysis(NSIDE, LMAX, rc[0])
    low = (m >= 10) & (l - m < 4)
    for b in range(2):
        assert _worst(got[b, 0][low], ref[0][low], floor) < bar
