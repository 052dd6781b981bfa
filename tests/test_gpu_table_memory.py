"""Tables that are made on first use and do not fit: the calls run without them
(the mixed mode, which has no such kernels at this size, reports DM_ENOMEM), the
plan holds nothing of an attempt that failed, and a later call makes them once
there is memory.  Bars: 1e-12 for FP64-class transforms, 2e-6 for mixed ones."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import alm_dev, dev, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1801_05358_gb300 import dmwf  # noqa: E402

NSIDE, LMAX = 128, 256


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _transforms(p, alm, maps):
    m = torch.zeros(tuple(maps.shape), dtype=torch.float64, device="cuda")
    a = torch.zeros(tuple(alm.shape) + (2,), dtype=torch.float64, device="cuda")
    p.alm2map(alm_dev(alm), m)
    p.map2alm(dev(maps), a)
    torch.cuda.synchronize()
    return m.cpu().numpy(), a.cpu().numpy().view(np.complex128)[..., 0]


# 0: nothing fits; 20 MB: the ring scratch does, its matrices and the Legendre digits do not
@pytest.mark.parametrize("prec", [dmwf.DM_FP64, dmwf.DM_FLOAT_FLOAT])
@pytest.mark.parametrize("limit", [0, 20_000_000])
def test_fp64_class_recovers(orc, prec, limit):
    B = 2
    alm, maps = W.random_alm(LMAX, B, 15), W.random_maps(NSIDE, B, 16)
    p = dmwf.Plan(NSIDE, LMAX, B)
    p.set_precision(prec)
    held = p.info()["workspace_bytes"]
    p.test_table_memory(limit)
    out = [_transforms(p, alm, maps)]
    assert p.info()["workspace_bytes"] == held
    p.test_table_memory()
    out.append(_transforms(p, alm, maps))
    assert p.info()["workspace_bytes"] > held
    p.close()
    for b in range(B):
        rm, ra = orc.alm2map(NSIDE, LMAX, alm[b]), orc.map2alm(NSIDE, LMAX, maps[b])
        for gm, ga in out:
            assert rel(gm[b], rm) < 1e-12 and rel(ga[b], ra) < 1e-12


def test_mixed_recovers(orc):
    B = 3
    alm, maps = W.random_alm(LMAX, B, 17), W.random_maps(NSIDE, B, 18)
    p = dmwf.Plan(NSIDE, LMAX, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    p.test_table_memory(0)
    for _ in range(2):
        with pytest.raises(dmwf.DmError) as ei:
            _transforms(p, alm, maps)
        assert ei.value.status == dmwf.DM_ENOMEM
    p.test_table_memory()
    gm, ga = _transforms(p, alm, maps)
    p.close()
    for b in range(B):
        assert rel(gm[b], orc.alm2map(NSIDE, LMAX, alm[b])) < 2e-6
        assert rel(ga[b], orc.map2alm(NSIDE, LMAX, maps[b])) < 2e-6
