"""The FP32 phases of the initial conditions (Box-Muller in pairs of FP32 numbers) against their FP64
values.

The logarithm is within 5.5e-11 of its value and the cosine within 6.2e-11 (the sine within 7e-12),
so a phase is within 9e-11 before its last rounding, 0.0015 units: at most 0.502 units off.  Their
rms errors (4.9e-12 and 6.3e-12) move a rounding in fewer than one in ten thousand."""
import numpy as np
import pytest

from tests.gpu_util import lib, to_dev, to_host, torch

pytestmark = pytest.mark.gpu


def _words():
    rng = np.random.default_rng(11)
    w = rng.integers(0, 2**32, (2_000_000, 2), dtype=np.uint64)
    edge = np.concatenate([np.arange(64), 2**32 - 1 - np.arange(64), (2**32 // 8) * np.repeat(np.arange(1, 8), 9) + np.tile(np.arange(-4, 5), 7),
                           (2.0**32 / np.sqrt(2.0)) + np.arange(-8, 9)]).astype(np.uint64)
    grid = np.stack([v.ravel() for v in np.meshgrid(edge, edge, indexing="ij")], axis=1)
    return np.concatenate([w, grid]).astype(np.uint32)


def test_phases_round_as_in_fp64():
    pm = lib()
    w = _words()
    out = torch.empty((len(w), 2), dtype=torch.float32, device="cuda")
    pm.pm_phase_check(to_dev(w), out)
    got = to_host(out).astype(np.float64)
    u = (w.astype(np.longdouble) + 0.5) / 2**32
    amp = np.sqrt(-np.log(u[:, 0]))
    # the angle's distance from the nearest quarter turn, exactly, so that sin and cos keep their digits
    k = np.rint(u[:, 1] * 4)
    x = (u[:, 1] * 4 - k) * (np.longdouble("1.57079632679489661923132169163975144"))
    s, c = np.sin(x), np.cos(x)
    k = k.astype(np.int64) % 4
    re = np.select([k == 0, k == 1, k == 2], [c, -s, -c], s) * amp
    im = np.select([k == 0, k == 1, k == 2], [s, c, -s], -c) * amp
    for exact, mine in ((re, got[:, 0]), (im, got[:, 1])):
        nearest = exact.astype(np.float32)
        unit = np.spacing(np.abs(nearest)).astype(np.longdouble)
        assert np.max(np.abs(mine - exact) / unit) < 0.502
        assert np.mean(mine != nearest.astype(np.float64)) < 1e-4
