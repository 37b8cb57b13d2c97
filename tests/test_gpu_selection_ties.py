"""The halo proxy's radix selection at its edges: ties at the threshold that are all taken, partly
taken or fill the field, values that share their leading digits, signed zeros and negative values,
the smallest and largest fractions, and unaligned fields.  Exact against the oracle's ranking (ties
by the lower index)."""
import numpy as np
import pytest

from oracle import stats
from tests.gpu_util import lib, to_host, torch

pytestmark = pytest.mark.gpu


def _fields(n, dt):
    rng = np.random.default_rng(n)
    g = rng.standard_normal((n, n, n))
    close = 1.0 + rng.integers(0, 40, (n, n, n)) * (2.0**-23 if dt == np.float32 else 2.0**-52)
    return {"gaussian": g, "integers": np.floor(2.0 * g), "constant": np.full((n, n, n), -0.25),
            "low bits": close, "negative": -np.abs(g) - 1.0, "tiny": g * 1e-40 if dt == np.float32 else g * 1e-310}


@pytest.mark.parametrize("prec,dt", [(0, np.float32), (1, np.float64)])
@pytest.mark.parametrize("n", [16, 32])
@pytest.mark.parametrize("fraction", [1e-9, 0.05, 0.5, 1.0])
def test_selection_matches_oracle(n, fraction, prec, dt):
    pm = lib()
    run = pm.PMRun(pm.make_config(n, n, 500.0, 0.02, 1.0, 10, precision=prec))
    for name, f in _fields(n, dt).items():
        f = f.astype(dt)
        for shift in (0, 1):  # an address off the four-value vectors
            buf = torch.empty(n**3 + shift, dtype=torch.float64 if prec else torch.float32, device="cuda")
            field = buf[shift:].view(n, n, n)
            field.copy_(torch.from_numpy(f))
            out = torch.full_like(buf, 7.0)[shift:].view(n, n, n)
            k = pm.pm_halo_proxy(run.ctx, out, field=field, fraction=fraction)
            mask = stats.top_fraction_mask(f, fraction)
            assert k == mask.sum(), name
            got = to_host(out)
            np.testing.assert_array_equal(got > got.min() if k < n**3 else np.ones_like(mask), mask, err_msg=name)
            np.testing.assert_allclose(got[mask], n**3 / k - 1.0, rtol=1e-6, atol=1e-12, err_msg=name)
