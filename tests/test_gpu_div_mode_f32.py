"""The FP32 per-mode divide of the spectral operators (quotient by the approximate reciprocal, one
correction from its remainder) against the correctly rounded division.

The approximate reciprocal is within 2 units (CUDA's bound for __fdividef), so the first quotient is
within 4, the remainder is exact, and the correction leaves an error of some 4 x 2^-21 units before
the last rounding: the result is the rounded quotient but where that lies within 2^-18 units of a
tie, i.e. but for 2^-17 of all operands, and is a neighbour of it there."""
import numpy as np
import pytest

from tests.gpu_util import lib, to_dev, to_host, torch

pytestmark = pytest.mark.gpu


def _check(a, d):
    pm = lib()
    a, d = np.asarray(a, dtype=np.float32), np.asarray(d, dtype=np.float32)
    out = torch.empty(a.size, dtype=torch.float32, device="cuda")
    pm.pm_div_mode_check_f32(to_dev(a), to_dev(d), out)
    got, want = to_host(out), a / d  # numpy: IEEE correctly rounded
    assert np.all(np.sign(got) == np.sign(want))
    ulps = np.abs(np.abs(got).view(np.int32) - np.abs(want).view(np.int32))
    assert ulps.max() <= 1
    return np.mean(ulps > 0)


def test_green_function_operands():
    # coef / (kf^2) over every |n|^2 of a 1024^3 mesh, boxes from 100 Mpc/h to 20 Gpc/h
    n2 = np.arange(1, 3 * 512**2 + 1)
    for box in (100.0, 2000.0, 5000.0, 20000.0):
        kf = 2 * np.pi / box
        for n in (64.0, 512.0):
            assert _check(np.full(n2.size, -1.5 * 0.31 / n**3 / kf**2), n2) < 2.0**-17


def test_constraint_denominators():
    r = np.random.default_rng(1)
    m = 1_000_000
    H = 10**r.uniform(np.log10(3e-5), np.log10(3e-4), m)
    dtau = 10**r.uniform(np.log10(5.0), np.log10(500.0), m)
    k = 10**r.uniform(np.log10(3e-4), np.log10(16.0), m)
    om = r.uniform(0.3, 1.0, m)
    d = k * k + 3 * H / dtau + 3 * H * H + 4.5 * H * H * om
    for a in (np.ones(m), -1.5 * H * H * om, 3 * H / dtau):
        assert _check(a, d) < 2.0**-17


def test_whole_range():
    r = np.random.default_rng(2)
    m = 2_000_000
    d = 2.0**r.uniform(-126, 126, m)
    a = d * 2.0**r.uniform(-40, 40, m) * r.choice([-1.0, 1.0], m)
    keep = (np.abs(a) > 2.0**-100) & (np.abs(a) < 2.0**127)
    assert _check(a[keep], d[keep]) < 2.0**-17
    pm = lib()
    out = torch.empty(3, dtype=torch.float32, device="cuda")
    pm.pm_div_mode_check_f32(torch.zeros(3, device="cuda"), torch.tensor([1e-30, 1.0, 1e30], device="cuda"), out)
    assert not to_host(out).any()
