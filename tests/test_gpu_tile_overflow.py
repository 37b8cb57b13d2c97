"""Deposit tiles in which cells pass 256 mass units, the range of their 32-bit fixed-point cells:
every particle of a Lagrangian block (16 x 16 x 32 mesh cells) is moved into one cell near the
block's centre, so a cell holds up to 8192 mass units.

The density is compared with the FP64 oracle's deposit of the same ticks.  Each of the N <= 8192
additions of a cell is off by half a quantum of 2^-24 at most, and the cell's value is of the
order of N, so the relative error stays below the FP32 rounding of the weights: 1e-6 relative L2,
the tolerance of the plain deposit."""
import numpy as np
import pytest

from oracle import cic
from tests.gpu_util import lib, rel_l2, to_dev, to_host, torch

pytestmark = pytest.mark.gpu


def _collapsed(np_side, n):
    """uint32 ticks: each block's particles in the cell nearest its centre, spread within it."""
    r = n // np_side
    i = np.arange(np_side)
    q = np.stack([v.ravel() for v in np.meshgrid(i, i, i, indexing="ij")])
    block = np.array([16 // r, 16 // r, 32 // r])[:, None]
    centre = (q // block * block + block // 2) * r  # mesh cells
    rng = np.random.default_rng(n + np_side)
    frac = centre + 0.5 + rng.uniform(0.05, 0.95, size=centre.shape)  # nodes sit at cell centres
    return np.floor(frac * (2.0**32 / n)).astype(np.int64).astype(np.uint32)


@pytest.mark.parametrize("np_side,n", [(64, 64), (128, 128), (32, 64), (64, 128), (16, 64)])
def test_dense_tiles_match_oracle(np_side, n):
    pm = lib()
    x = _collapsed(np_side, n)
    # a huge box and a short step: the update's drift is a small fraction of a cell
    run = pm.PMRun(pm.make_config(np_side, n, 1.0e5, 0.5, 0.501, 2))
    pm.pm_set_particles(run.ctx, to_dev(x), torch.zeros((3, np_side**3), dtype=torch.float32, device="cuda"))
    want = cic.density_contrast(x, n)
    assert want.max() > 500.0
    assert rel_l2(to_host(run.density()), want) < 1e-6
    # the density the fused update leaves behind, through the spectrum of it
    run.step(1)
    moved = to_host(run.particles()[0]).view(np.uint32)
    after = cic.density_contrast(moved, n)
    assert after.max() > 500.0
    edges = np.array([1.0, 2.0, 4.0, 8.0, n / 2.0])
    got = run.power(edges)[1]
    want_p = run.power(edges, field=to_dev(after.astype(np.float32)))[1]
    # FP32 rounds the density relative to its dense cells, evenly over the modes, and the periodic
    # clumps leave the lowest modes empty: relative to the spectrum's largest value
    assert np.max(np.abs(got - want_p)) < 2e-6 * np.max(want_p)
