"""The stateless particle operators on the smallest meshes they take (2 and 4 cells a side), whose
z rows hold no group of four cells or exactly one.  Against the FP64 oracle with the tolerances of
the plain tests (FP32 1e-6, FP64 1e-14 relative L2; keys and order exact); the cells beside the mesh
stay as they were."""
import numpy as np
import pytest

from oracle import cic
from tests.gpu_util import lib, rel_l2, to_dev, to_host, torch

pytestmark = pytest.mark.gpu
FP32, FP64 = 0, 1
TOL = {FP32: 1e-6, FP64: 1e-14}


def _points(n, prec):
    rng = np.random.default_rng(n)
    axis = np.concatenate([(np.arange(n) + 0.5) / n, np.arange(n) / n, [2.0**-40, 0.25 / n, 1.0 - 2.0**-32],
                           rng.uniform(size=64)])
    x = rng.choice(axis, size=(3, 1501))
    return x if prec == FP64 else np.floor(x * 2.0**32).astype(np.uint64).astype(np.uint32)


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("n", [2, 4])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_operators_match_oracle(n, prec, shift):
    pm = lib()
    xs = _points(n, prec)
    count = xs.shape[1]
    x = to_dev(xs)
    dt = torch.float64 if prec else torch.float32
    whole = torch.zeros(n**3 + shift + 8, dtype=dt, device="cuda")
    pm.pm_cic_deposit(x, count, prec, n, 1.0, whole[shift:])
    got = to_host(whole)
    assert rel_l2(got[shift:shift + n**3].reshape(n, n, n), cic.deposit(xs, n, 1.0)) < TOL[prec]
    assert not got[:shift].any() and not got[shift + n**3:].any()
    f = np.random.default_rng(17 + n).standard_normal((n, n, n)).astype(np.float64 if prec else np.float32)
    field = torch.full((n**3 + shift + 8,), float("nan"), dtype=dt, device="cuda")
    field[shift:shift + n**3].copy_(torch.from_numpy(f.ravel()))
    out = torch.empty(count, dtype=dt, device="cuda")
    pm.pm_cic_interp(field[shift:], n, x, count, prec, out)
    assert rel_l2(to_host(out), cic.interpolate(f.astype(np.float64), xs)) < TOL[prec]
    keys, order = (torch.empty(count, dtype=torch.int32, device="cuda") for _ in range(2))
    scratch = torch.empty(pm.pm_cell_sort_scratch_size(count, n), dtype=torch.uint8, device="cuda")
    pm.pm_cell_sort(x, count, prec, n, keys, order, scratch)
    np.testing.assert_array_equal(to_host(keys).astype(np.int64), cic.cell_keys(xs, n))
    np.testing.assert_array_equal(to_host(order).astype(np.int64), cic.cell_order(xs, n))
