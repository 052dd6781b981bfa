"""The mixed mode's FP32 Legendre kernels where no digit table is kept whole and
with the tensor cores off: any size and batch, from tables kept for the life of
the plan; slabs of digits, made again in each call, only where those do not fit.
In the FP64-class modes one right-hand side without a whole table runs the
recurrence kernels.  Bars: 2e-6 for single mixed transforms, 1e-12 for
FP64-class ones, 1e-5 for a mixed solve."""
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


def _check(orc, p, nside, lmax, B, bar):
    alm, maps = W.random_alm(lmax, B, 88), W.random_maps(nside, B, 89)
    m = torch.zeros((B, 3, 12 * nside * nside), dtype=torch.float64, device="cuda")
    a = torch.zeros((B, 3, alm.shape[-1], 2), dtype=torch.float64, device="cuda")
    p.alm2map(alm_dev(alm), m)
    p.map2alm(dev(maps), a)
    torch.cuda.synchronize()
    ga = a.cpu().numpy().view(np.complex128)[..., 0]
    for b in sorted({0, B // 2, B - 1}):
        assert rel(m[b].cpu().numpy(), orc.alm2map(nside, lmax, alm[b])) < bar
        assert rel(ga[b], orc.map2alm(nside, lmax, maps[b])) < bar


def _table_bytes(nside, lmax):
    return 12 * ((lmax + 1) * (lmax + 2) // 2) * ((2 * nside + 3) // 4 * 4)


# batches of every width of the kernels (1, 2, 4 right-hand sides a thread or
# block), ring pairs and multipoles off the tiles' edges; slabs of one order
@pytest.mark.parametrize("way", ["slabs", "no tensor cores"])
@pytest.mark.parametrize("nside,lmax,B", [(101, 250, 1), (129, 256, 2), (128, 255, 3), (97, 300, 5), (64, 200, 8), (100, 260, 14)])
def test_mixed_without_a_whole_table(orc, nside, lmax, B, way):
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    if way == "slabs":
        if B == 8:
            pytest.skip("a tensor-core batch")
        p.set_ff_slab_bytes(1)
    else:
        p.set_tensor_cores(False)
    held = p.info()["workspace_bytes"]
    _check(orc, p, nside, lmax, B, 2e-6)
    assert p.info()["workspace_bytes"] - held == _table_bytes(nside, lmax)
    p.close()


def test_mixed_slabs_where_the_tables_do_not_fit(orc):
    nside, lmax, B = 128, 256, 3
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    p.set_ff_slab_bytes(2_000_000)
    p.test_table_memory(_table_bytes(nside, lmax) - 1)
    _check(orc, p, nside, lmax, B, 2e-6)
    p.close()


@pytest.mark.parametrize("prec", [dmwf.DM_FP64, dmwf.DM_FLOAT_FLOAT])
def test_one_right_hand_side_in_slabs(orc, prec):
    nside, lmax = 60, 128  # below the size of the ring products: no other table is made
    p = dmwf.Plan(nside, lmax, 1)
    p.set_precision(prec)
    p.set_ff_slab_bytes(1)
    held = p.info()["workspace_bytes"]
    _check(orc, p, nside, lmax, 1, 1e-12)
    assert p.info()["workspace_bytes"] == held
    p.close()


def test_mixed_solve_in_slabs(orc):
    wl = W.make_workload("nside16", [0, 1, 2], nside=64, lmax=128)
    d = np.stack([wl.data([orc.alm2map(wl.nside, wl.lmax, a)])[0] for a in wl.alm_true])
    lam = W.lambda_schedule(100.0, 3)
    p = make_plan(wl, 3, lambda0=100.0, n_levels=3, iters_per_level=3, check_every=4)
    p.set_precision(dmwf.DM_MIXED_FP32)
    p.set_ff_slab_bytes(100_000)
    s = torch.zeros((3, 3, wl.npix), dtype=torch.float64, device="cuda")
    p.wiener_filter(dev(d), s)
    p.close()
    for b in range(3):
        ref = orc.dm_solve(wl.nside, wl.lmax, wl.cl, wl.sigma, wl.mask, d[b], lam, forced_iters=[3, 3, 3])
        assert rel(s[b].cpu().numpy(), ref["s"]) < 1e-5


# The default choice of the analysis: four right-hand sides a block from eight on
# where that fills the chip (the last block with one to four), two or one else;
# ring pairs within one warp's pass and in several, odd rows at the end.
@pytest.mark.parametrize("nside,lmax,B", [(2, 4, 12), (23, 60, 12), (64, 190, 12), (33, 67, 20), (64, 128, 14),
                                          (64, 128, 19), (33, 70, 17), (16, 33, 4), (16, 33, 17), (16, 33, 50)])
def test_mixed_batches(orc, nside, lmax, B):
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    _check(orc, p, nside, lmax, B, 2e-6)
    p.close()


# The anchors' digits are made first in a solve: room for them is not asked for again.
def test_tables_beside_the_anchors_digits():
    nside, lmax, B = 128, 256, 3
    npix = 12 * nside * nside
    p = dmwf.Plan(nside, lmax, B)
    p.set_precision(dmwf.DM_MIXED_FP32)
    p.set_ring_radix(3)
    p.set_diagnostics(False)
    p.set_ff_slab_bytes(2_000_000)
    p.set_noise_mask(np.full((3, npix), 0.5), np.ones(npix, np.uint8))
    cl = np.zeros((4, lmax + 1))
    cl[:3, 2:] = 1.0 / np.arange(2, lmax + 1) ** 2.0
    p.set_spectra(cl)
    p.set_schedule(lambda0=10.0, n_levels=1, iters_per_level=2, check_every=2)
    p.test_table_memory(_table_bytes(nside, lmax))
    held = p.info()["workspace_bytes"]
    d = dev(W.random_maps(nside, B, 90))
    p.wiener_filter(d, torch.zeros_like(d))
    assert p.info()["workspace_bytes"] - held > _table_bytes(nside, lmax)
    p.close()
