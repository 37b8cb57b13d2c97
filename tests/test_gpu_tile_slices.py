"""Lattices so small that a deposit block is shared by several CTAs (64^3 meshes): clumped particles
are still summed in fixed point, each slice's part of a cell being rounded once.

A cell of eight slices' parts is rounded by half a unit of each part, and by half a unit of the
running sum at each of their additions: at most 2^-24 (1 + 1/8 + 2/8 + ... + 8/8) of its value,
3.3e-7.  Added particle by particle the same lattice was off by 9.1e-7 (64^3) and 3.1e-7 (32^3)
relative L2, where the sums of parts are off by their roundings' rms, some 6e-8; the bound is
2^-22."""
import numpy as np
import pytest

from oracle import cic
from tests.gpu_util import lib, rel_l2, to_dev, to_host, torch
from tests.test_gpu_tile_overflow import _collapsed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_side", [64, 32, 16])
def test_density_of_clumps(np_side):
    pm = lib()
    n = 64
    x = _collapsed(np_side, n)
    run = pm.PMRun(pm.make_config(np_side, n, 1.0e5, 0.5, 0.501, 2))
    pm.pm_set_particles(run.ctx, to_dev(x), torch.zeros((3, np_side**3), dtype=torch.float32, device="cuda"))
    for _ in range(3):
        assert rel_l2(to_host(run.density()), cic.density_contrast(x, n)) < 2.0**-22


@pytest.mark.parametrize("np_side", [64, 32, 16])
@pytest.mark.parametrize("moved", [0, 3, 11, 30])
def test_slices_that_fill_any_planes(np_side, moved):
    """Particles displaced by whole cells along x: within their slice's planes, across the block's,
    half and wholly out of its box."""
    pm = lib()
    n, r = 64, 64 // np_side
    i = np.arange(np_side)
    q = np.stack([v.ravel() for v in np.meshgrid(i, i, i, indexing="ij")]) * r
    rng = np.random.default_rng(moved)
    x = np.floor((q + rng.uniform(0, r, q.shape)) * (2.0**32 / n)).astype(np.int64)
    x[0] += rng.integers(-moved, moved + 1, x.shape[1]) * (2**32 // n)
    x = (x % 2**32).astype(np.uint32)
    run = pm.PMRun(pm.make_config(np_side, n, 1.0e5, 0.5, 0.501, 2))
    pm.pm_set_particles(run.ctx, to_dev(x), torch.zeros((3, np_side**3), dtype=torch.float32, device="cuda"))
    assert rel_l2(to_host(run.density()), cic.density_contrast(x, n)) < 1e-6
    edges = np.array([1.0, 4.0, 16.0, 32.0])
    run.step(1)
    got = run.power(edges)[1]  # of the density that the update left
    after = cic.density_contrast(to_host(run.particles()[0]).view(np.uint32), n)
    want = run.power(edges, field=to_dev(after.astype(np.float32)))[1]
    assert np.max(np.abs(got / want - 1)) < 1e-5
