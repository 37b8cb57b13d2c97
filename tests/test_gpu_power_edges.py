"""P(k) whose last edge stops below, at or beyond the Nyquist sphere: the transform leaves out the
kz planes and the binning pass the columns that no bin reaches.  Against the FP64 oracle, with the
tolerances of the full range (FP32 2e-6, FP64 1e-12; mode counts exact)."""
import numpy as np
import pytest

import inputs
from oracle import stats
from tests.gpu_util import lib, to_dev

pytestmark = pytest.mark.gpu
FP32, FP64 = 0, 1
TOL = {FP32: 2e-6, FP64: 1e-12}
EDGES = ([0.25, 0.5], [1.0, 2.5], [0.5, 1.0, 2.0, 5.0**0.5], [1.0, 3.0, 7.0, 8.0], [2.0, 9.0, 15.999, 16.0],
         [1.0, 12.0, 40.0])


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("n", [16, 32, 64])
@pytest.mark.parametrize("edges", EDGES)
def test_power_matches_oracle_for_any_last_edge(edges, n, prec):
    pm = lib()
    dt = np.float64 if prec == FP64 else np.float32
    f = inputs.gaussian_field(500 + n, n).astype(dt)
    g = inputs.lognormal_field(600 + n, n, sigma=0.5).astype(dt)
    run = pm.PMRun(pm.make_config(n, n, 700.0, 0.02, 1.0, 10, precision=prec))
    for second in (None, g):
        k, p, nm = run.power(np.array(edges), field=to_dev(f), field2=None if second is None else to_dev(second))
        kr, pr, nr = stats.power_spectrum(f.astype(np.float64), 700.0, np.array(edges),
                                          delta2=None if second is None else second.astype(np.float64))
        np.testing.assert_array_equal(nm, nr)
        ok = nr > 0
        np.testing.assert_allclose(k[ok], kr[ok], rtol=1e-12)
        # cross spectra cancel: relative to the spectra's scale
        scale = np.abs(pr[ok]) if second is None else np.sqrt(
            stats.power_spectrum(f.astype(np.float64), 700.0, np.array(edges))[1][ok] *
            stats.power_spectrum(second.astype(np.float64), 700.0, np.array(edges))[1][ok])
        assert np.all(np.abs(p[ok] - pr[ok]) <= TOL[prec] * scale)
        assert np.all(np.isnan(p[~ok]))
