"""Rounding error of the FP32 transforms of white noise against 64 bits, per mesh side.

The bounds are the relative L2 errors of transforms of eight elements a thread (three radix-8 stages
at 512), measured on white noise and rounded up in the third digit: 1.36, 1.48, 1.62, 1.73 and
1.85e-7 forward, 1.37, 1.49, 1.62, 1.73 and 1.85e-7 inverse, plus 1% for the spread between fields
(the error averages over at least 2^14 modes).  Two stages with rounded cosines and sines as the
constants of their butterflies exceed them from 64 up (1.52, 1.65, 1.80, 1.97e-7)."""
import pytest

from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu

BOUNDS = {32: 1.37e-7, 64: 1.49e-7, 128: 1.62e-7, 256: 1.74e-7, 512: 1.85e-7}


@pytest.mark.parametrize("n", sorted(BOUNDS))
def test_fft_error_of_white_noise(n):
    pm = lib()
    g = torch.Generator("cuda")
    g.manual_seed(n)
    f = torch.randn((n, n, n), generator=g, device="cuda")
    spec = torch.empty((n // 2 + 1, n, n), dtype=torch.complex64, device="cuda")
    pm.pm_fft_r2c(f, spec, n, pm.PM_FP32_FIXED)
    want = torch.fft.rfftn(f.double())
    err = (spec.to(torch.complex128) - want.permute(2, 0, 1)).norm() / want.norm()
    assert float(err) < 1.01 * BOUNDS[n]
    half = want.permute(2, 0, 1).to(torch.complex64).contiguous()
    back = torch.fft.irfftn(half.to(torch.complex128).permute(1, 2, 0), s=(n, n, n), norm="forward")
    out = torch.empty_like(f)
    pm.pm_fft_c2r(half, out, n, pm.PM_FP32_FIXED)
    assert float((out.double() - back).norm() / back.norm()) < 1.01 * BOUNDS[n]
