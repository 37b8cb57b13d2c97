"""Deposit tiles whose cells pass 2^32 quanta (256 mass units), in every instance of the second
accumulation (both force gradients, every tile depth, batches): a cell's remainder below 256 units
and its wraps, all at once, are added to the mesh.

A cell of one dense tile and a little from its neighbour is so rounded at most twice at its own
unit, by the wraps and by the neighbour's part where that comes last, and at a quarter of it or less
before that: an rms error of at most sqrt((1 + 1 + 1/16 + 1/64) / 12) = 0.416 units, with a spread
of 1.4% over 1024 cells; the bound is 0.44.  Wraps added one by one round at every doubling of the
sum: 0.48 and more.

Parity of the densities with the tolerances of tests/test_gpu_tile_overflow.py."""
import numpy as np
import pytest

from oracle import cic
from tests.gpu_util import lib, min_image, positions_box_units, rel_l2, ticks_to_host, to_dev, to_host, torch
from tests.test_gpu_tile_overflow import _collapsed

pytestmark = pytest.mark.gpu
EDGES64 = np.array([1.0, 2.0, 4.0, 8.0, 32.0])


@pytest.mark.parametrize("keep", [0.8, 0.6])
def test_rounding_of_dense_cells(keep):
    pm = lib()
    n = 128  # one cell a particle, tiles of 16 x 16 x 32
    i = np.arange(n)
    q = np.stack([v.ravel() for v in np.meshgrid(i, i, i, indexing="ij")])
    tile = q // np.array([16, 16, 32])[:, None]
    # of two tiles along x the left one has most of its particles in one cell at their border, the
    # right one 16 there and the rest on the lattice
    left = tile[0] % 2 == 0
    guest = ~left & (q[0] % 16 == 0) & (q[1] % 16 < 4) & (q[2] % 32 < 4)
    border = np.stack([tile[0] // 2 * 32 + 15, tile[1] * 16 + 8, tile[2] * 32 + 8])
    rng = np.random.default_rng(int(10 * keep))
    clump = (left & (rng.uniform(size=q.shape[1]) < keep)) | guest
    x = np.where(clump, border + 0.5 + rng.uniform(0.02, 0.98, q.shape), q + 0.75)
    x = np.floor(x * (2.0**32 / n)).astype(np.int64).astype(np.uint32)
    want = cic.density_contrast(x, n)
    dense = want > 300.0
    assert dense.sum() == 1024
    run = pm.PMRun(pm.make_config(n, n, 1.0e5, 0.5, 0.501, 2))
    pm.pm_set_particles(run.ctx, to_dev(x), torch.zeros((3, n**3), dtype=torch.float32, device="cuda"))
    unit = np.spacing(want[dense].astype(np.float32)).astype(np.float64)
    err = (to_host(run.density()).astype(np.float64)[dense] - want[dense]) / unit
    assert np.sqrt(np.mean(err**2)) < 0.44


def _check_steps(run, x, n):
    """The density of dense tiles, and the one that the update leaves behind."""
    want = cic.density_contrast(x, n)
    assert want.max() > 500.0
    assert rel_l2(to_host(run.density()), want) < 1e-6
    run.step(1)
    after = cic.density_contrast(to_host(run.particles()[0]).view(np.uint32), n)
    assert after.max() > 500.0
    got = run.power(EDGES64)[1]
    want_p = run.power(EDGES64, field=to_dev(after.astype(np.float32)))[1]
    assert np.max(np.abs(got - want_p)) < 2e-6 * np.max(want_p)


@pytest.mark.parametrize("np_side,n", [(64, 64), (128, 128), (32, 64), (16, 64)])
def test_first_order_gradient(np_side, n):
    pm = lib()
    x = _collapsed(np_side, n)
    run = pm.PMRun(pm.make_config(np_side, n, 1.0e5, 0.5, 0.501, 2, gradient=pm.PM_GRAD_FD1))
    pm.pm_set_particles(run.ctx, to_dev(x), torch.zeros((3, np_side**3), dtype=torch.float32, device="cuda"))
    _check_steps(run, x, n)


# tiles of depth 4, 8 and 16 on 64^3 meshes (one run alone takes depth 2)
@pytest.mark.parametrize("np_side", [64, 32, 16])
@pytest.mark.parametrize("nreal", [2, 3, 5])
def test_batches(np_side, nreal):
    pm = lib()
    n, box = 64, 1.0e5
    x = _collapsed(np_side, n)
    cfg = pm.make_config(np_side, n, box, 0.5, 0.501, 2)
    batch = pm.PMBatch(cfg, boxes=[box] * nreal)
    batch.ic(list(range(nreal)))
    run = pm.PMRun(cfg)
    # every realisation is another density: its clumps moved within their cells
    xs = [x + np.uint32(r * (2**32 // n) // 128) for r in range(nreal)]
    for r in range(nreal):
        xr, pr = batch.particles(r)
        xr.copy_(to_dev(xs[r]))
        pr.zero_()
    power = batch.power(EDGES64)[1]
    batch.step(2)
    for r in range(nreal):
        pm.pm_set_particles(run.ctx, to_dev(xs[r]), torch.zeros((3, np_side**3), dtype=torch.float32, device="cuda"))
        field = to_dev(cic.density_contrast(xs[r], n).astype(np.float32))
        want_p = run.power(EDGES64, field=field)[1]
        assert np.max(np.abs(power[r] - want_p)) < 2e-6 * np.max(want_p)
        # two steps (the second's forces come from the density that the first's update left)
        run.step(2)
        (xb, pb), (xr, pr) = batch.particles(r), run.particles()
        moved = [min_image(positions_box_units(ticks_to_host(v)) - positions_box_units(xs[r])) for v in (xb, xr)]
        assert rel_l2(*moved) < 1e-5
        assert rel_l2(to_host(pb), to_host(pr)) < 1e-5
