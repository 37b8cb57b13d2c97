"""FP32 deposit with a mass that is infinite or not a number, or whose products overflow: the eight
cells of a particle take what the products give, every other cell stays 0 (a row's two cells may be
added as part of an aligned group of four)."""
import numpy as np
import pytest

from oracle import cic
from tests.gpu_util import lib, to_dev, to_host, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mass", [float("inf"), float("-inf"), float("nan"), 3.0e38])
@pytest.mark.parametrize("shift", [0, 1])
def test_cells_beside_a_particle_stay_zero(mass, shift):
    pm = lib()
    n = 16
    rng = np.random.default_rng(3)
    # one particle in every fourth cell along each axis, off the nodes: no two touch the same cell
    q = np.stack([v.ravel() for v in np.meshgrid(*[np.arange(0, n, 4)] * 3, indexing="ij")])
    for z in range(4):  # every place in a group of four
        at = q + np.array([1, 2, z])[:, None]
        x = np.floor((at + 0.5 + rng.uniform(0.2, 0.8, at.shape)) * (2.0**32 / n)).astype(np.int64).astype(np.uint32)
        rho = torch.zeros(n**3 + shift, dtype=torch.float32, device="cuda")[shift:]
        pm.pm_cic_deposit(to_dev(x), x.shape[1], 0, n, mass, rho)
        got = to_host(rho).reshape(n, n, n)
        weights = cic.deposit(x, n, 1.0)
        touched = weights > 0
        assert touched.sum() == 8 * x.shape[1]
        assert not got[~touched].any()
        if np.isfinite(mass):
            np.testing.assert_allclose(got[touched], mass * weights[touched], rtol=1e-6)
        else:
            assert np.array_equal(np.isnan(got[touched]), np.isnan(mass * weights[touched]))
            assert not np.isfinite(got[touched]).any()
