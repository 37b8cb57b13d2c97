"""GPU parity of the FFT passes at every transform length up to 512: each length has its own
split into register stages, row layout and launch shape.  Expected values: torch's FP64
transforms of the same seeded mesh.  Tolerances as for the smaller meshes (FP32: a few times
eps log2 n^3, FP64 likewise)."""
import pytest

from tests.gpu_util import empty_spec, lib, torch

pytestmark = pytest.mark.gpu
FP32, FP64 = 0, 1
TOL = {FP32: 2e-6, FP64: 1e-13}


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("n", [16, 32, 64, 128, 256, 512])
def test_transforms_match_fp64(n, prec):
    pm = lib()
    dt = torch.float64 if prec == FP64 else torch.float32
    f = torch.randn((n, n, n), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda", dtype=dt)
    ref = torch.fft.rfftn(f.double())
    spec = empty_spec(n, prec == FP64)
    pm.pm_fft_r2c(f, spec, n, prec)
    got = torch.view_as_complex(spec.reshape(n // 2 + 1, n, n, 2)).permute(1, 2, 0)
    assert float(torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)) < TOL[prec]
    # the inverse of a spectrum that is not the transform's own output
    ref = ref * 0.5
    spec = torch.view_as_real(ref.permute(2, 0, 1).contiguous()).to(dt).contiguous()
    out = torch.empty_like(f)
    pm.pm_fft_c2r(spec, out, n, prec)
    want = f.double() * (0.5 * n**3)
    assert float(torch.linalg.vector_norm(out - want) / torch.linalg.vector_norm(want)) < TOL[prec]
