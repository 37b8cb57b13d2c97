"""The particle operators at the edges of their vector and bit forms: positions on and next to mesh
nodes, in the first and last half cell, at 0 and just below 1, meshes whose address is off the
16-byte vectors, cells of 1 to 40 particles.  Against the FP64 oracle with the tolerances of the
plain tests (deposit and interpolation FP32 1e-6, FP64 1e-14 relative L2; keys and order exact)."""
import numpy as np
import pytest

import inputs
from oracle import cic
from tests.gpu_util import lib, rel_l2, to_dev, to_host, torch

pytestmark = pytest.mark.gpu
FP32, FP64 = 0, 1
TOL = {FP32: 1e-6, FP64: 1e-14}


def _points(n, prec):
    rng = np.random.default_rng(n)
    node = (np.arange(n) + 0.5) / n
    tiny = 2.0**-40
    axis = np.concatenate([node, np.maximum(node - tiny, 0), node + tiny, np.arange(n) / n,
                           [0.0, tiny, 2.0**-60, 0.25 / n, 0.75 / n, 1.0 - 2.0**-53, 1.0 - 2.0**-32, 1.0 - 0.25 / n]])
    x = rng.choice(axis, size=(3, 4001))
    crowd = np.repeat((rng.integers(0, n, (3, 40)) + 0.3) / n, np.arange(1, 41), axis=1)
    x = np.concatenate([x, crowd], axis=1)
    return x if prec == FP64 else np.floor(x * 2.0**32).astype(np.uint64).astype(np.uint32)


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("n", [8, 16, 64])
@pytest.mark.parametrize("shift", [0, 1])
def test_operators_match_oracle(n, prec, shift):
    pm = lib()
    xs = _points(n, prec)
    count = xs.shape[1]
    x = to_dev(xs)
    dt = torch.float64 if prec else torch.float32
    rho = torch.zeros(n**3 + shift, dtype=dt, device="cuda")[shift:]
    pm.pm_cic_deposit(x, count, prec, n, 1.0, rho)
    assert rel_l2(to_host(rho).reshape(n, n, n), cic.deposit(xs, n, 1.0)) < TOL[prec]
    f = inputs.gaussian_field(n, n).astype(np.float64 if prec else np.float32)
    field = torch.empty(n**3 + shift, dtype=dt, device="cuda")[shift:]
    field.copy_(torch.from_numpy(f.ravel()))
    out = torch.empty(count, dtype=dt, device="cuda")
    pm.pm_cic_interp(field, n, x, count, prec, out)
    assert rel_l2(to_host(out), cic.interpolate(f.astype(np.float64), xs)) < TOL[prec]
    keys, order = (torch.empty(count, dtype=torch.int32, device="cuda") for _ in range(2))
    scratch = torch.empty(pm.pm_cell_sort_scratch_size(count, n), dtype=torch.uint8, device="cuda")
    pm.pm_cell_sort(x, count, prec, n, keys, order, scratch)
    np.testing.assert_array_equal(to_host(keys).astype(np.int64), cic.cell_keys(xs, n))
    np.testing.assert_array_equal(to_host(order).astype(np.int64), cic.cell_order(xs, n))


@pytest.mark.parametrize("np_side,n", [(16, 16), (32, 32), (16, 32), (64, 64)])
def test_fp64_context_density_matches_oracle(np_side, n):
    pm = lib()
    x = inputs.ticks_to_fractions(inputs.lattice_order_ticks(5 + n, np_side, 1.5, n_mesh=n, tail_fraction=0.02))
    run = pm.PMRun(pm.make_config(np_side, n, 500.0, 0.1, 1.0, 4, precision=FP64))
    pm.pm_set_particles(run.ctx, to_dev(x), torch.zeros((3, np_side**3), dtype=torch.float64, device="cuda"))
    assert rel_l2(to_host(run.density()), cic.density_contrast(x, n)) < 1e-13
