"""Rounding error of the FP64 transforms against extended precision, in the manner of
tests/test_gpu_fft_error.py: the bounds are the relative L2 errors of the three-stage transforms of
eight elements a thread.  Whole meshes of white noise (2.75e-16 at 32, 3.32e-16 at 64; there and
back 3.65 and 4.19), and for longer sides white noise on the line of one axis, whose transforms
along the other two are exact (rms over the axes and twelve lines each: 2.02e-16 at 128, 2.32 at
256, 2.51 at 512).  1% for the spread."""
import numpy as np
import pytest

from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu
fft = pytest.importorskip("scipy.fft")
WHOLE = {32: (2.75e-16, 3.65e-16), 64: (3.32e-16, 4.19e-16)}
AXIS = {128: 2.02e-16, 256: 2.32e-16, 512: 2.51e-16}


def _forward(f):
    pm = lib()
    n = f.shape[0]
    spec = torch.empty((n // 2 + 1, n, n), dtype=torch.complex128, device="cuda")  # [kz][kx][ky]
    pm.pm_fft_r2c(f, spec, n, pm.PM_FP64)
    return spec


def _rel(got, want):
    return float(np.sqrt(np.sum(np.abs(got - want)**2) / np.sum(np.abs(want)**2)))


@pytest.mark.parametrize("n", sorted(WHOLE))
def test_whole_meshes(n):
    pm = lib()
    f = np.random.default_rng(n + 7).standard_normal((n, n, n)).astype(np.float32).astype(np.float64)
    spec = _forward(torch.from_numpy(f).cuda())
    want = fft.rfftn(f.astype(np.longdouble)).transpose(2, 0, 1)
    assert _rel(spec.cpu().numpy(), want) < 1.01 * WHOLE[n][0]
    back = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
    pm.pm_fft_c2r(spec, back, n, pm.PM_FP64)
    assert _rel(back.cpu().numpy() / np.longdouble(n)**3, f) < 1.01 * WHOLE[n][1]


@pytest.mark.parametrize("n", sorted(AXIS))
def test_one_axis(n):
    f = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
    err = []
    for axis in range(3):
        line = tuple(slice(None) if a == axis else 0 for a in range(3))
        for seed in range(12):
            g = np.random.default_rng(1000 * n + 12 * axis + seed).standard_normal(n).astype(np.float32).astype(np.float64)
            f[line] = torch.from_numpy(g).cuda()
            spec = _forward(f)
            got = (spec[:, 0, 0] if axis == 2 else spec[0, :, 0] if axis == 0 else spec[0, 0, :]).cpu().numpy()
            err.append(_rel(got, fft.rfft(g.astype(np.longdouble)) if axis == 2 else fft.fft(g.astype(np.longdouble))))
        f[line] = 0.0
    assert np.sqrt(np.mean(np.square(err))) < 1.01 * AXIS[n]
