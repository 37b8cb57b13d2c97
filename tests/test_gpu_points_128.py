"""The particle operators on a 128^3 mesh, the first size whose cells do not all run at once: buckets
of 1 to 40 particles in the sort that keeps 8 in registers, FP64 positions in the first cell (bases
n - 1 and 0) and beyond, and the FP64 density of a 128^3 lattice, whose particles are deposited in
rows.  Tolerances of the plain tests (FP32 1e-6, FP64 1e-14 relative L2; keys and order exact)."""
import numpy as np
import pytest

import inputs
from oracle import cic
from tests.gpu_util import lib, rel_l2, to_dev, to_host, torch

pytestmark = pytest.mark.gpu
FP32, FP64 = 0, 1
TOL = {FP32: 1e-6, FP64: 1e-14}


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_operators_match_oracle(prec):
    pm = lib()
    n = 128
    rng = np.random.default_rng(prec)
    crowd = np.repeat((rng.integers(0, n, (3, 160)) + 0.3) / n, np.tile(np.arange(1, 41), 4), axis=1)
    first = rng.choice([0.0, 2.0**-70, 0.2 / n, 0.5 / n - 2.0**-40, 0.5 / n, 0.75 / n, 1.0 / n - 2.0**-40, 1.0 / n, 1.5 / n],
                       size=(3, 2000))
    x = rng.permutation(np.concatenate([crowd, first, rng.uniform(size=(3, 3000))], axis=1), axis=1)
    xs = x if prec == FP64 else np.floor(x * 2.0**32).astype(np.uint64).astype(np.uint32)
    count, dt = xs.shape[1], torch.float64 if prec else torch.float32
    dev = to_dev(xs)
    rho = torch.zeros(n**3, dtype=dt, device="cuda")
    pm.pm_cic_deposit(dev, count, prec, n, 1.0, rho)
    assert rel_l2(to_host(rho).reshape(n, n, n), cic.deposit(xs, n, 1.0)) < TOL[prec]
    f = rng.standard_normal((n, n, n)).astype(np.float64 if prec else np.float32)
    out = torch.empty(count, dtype=dt, device="cuda")
    pm.pm_cic_interp(to_dev(f), n, dev, count, prec, out)
    assert rel_l2(to_host(out), cic.interpolate(f.astype(np.float64), xs)) < TOL[prec]
    keys, order = (torch.empty(count, dtype=torch.int32, device="cuda") for _ in range(2))
    scratch = torch.empty(pm.pm_cell_sort_scratch_size(count, n), dtype=torch.uint8, device="cuda")
    pm.pm_cell_sort(dev, count, prec, n, keys, order, scratch)
    np.testing.assert_array_equal(to_host(keys).astype(np.int64), cic.cell_keys(xs, n))
    np.testing.assert_array_equal(to_host(order).astype(np.int64), cic.cell_order(xs, n))


def test_fp64_rows_match_oracle():
    pm = lib()
    n = 128
    x = inputs.ticks_to_fractions(inputs.lattice_order_ticks(7, n, 1.5, n_mesh=n, tail_fraction=0.02))
    run = pm.PMRun(pm.make_config(n, n, 500.0, 0.1, 1.0, 4, precision=FP64))
    pm.pm_set_particles(run.ctx, to_dev(x), torch.zeros((3, n**3), dtype=torch.float64, device="cuda"))
    assert rel_l2(to_host(run.density()), cic.density_contrast(x, n)) < 1e-13
