"""Batches larger than what one launch takes (128 seeds or scales by value, 65535 / 64 rows of the z
passes), and boxes whose tick scale rounds differently by another order of its operations: every
realisation has the particles of the single run with its box and seed, bit for bit, and its P(k)."""
import numpy as np
import pytest

from tests.gpu_util import lib, to_host, torch

pytestmark = pytest.mark.gpu
A_I, A_F = 0.9, 1.0


def _pair(v):
    """A double as the pair of FP32 numbers nearest it."""
    h = np.float32(v)
    return h, np.float32(v - np.float64(h))


def _single(pm, np_side, n, box, seed):
    run = pm.PMRun(pm.make_config(np_side, n, box, A_I, A_F, 4))
    run.ic(seed=seed)
    return run


def test_ticks_of_any_box_are_the_single_runs():
    pm = lib()
    np_side, n = 64, 64
    D = pm.pm_linear_power(pm.make_config(np_side, n, 100.0, A_I, A_F, 4), A_I, np.array([0.1]))[1]
    rng = np.random.default_rng(2)
    boxes = [b for b in rng.uniform(40.0, 160.0, 4000) if _pair(D * 2.0**32 / b) != _pair(D * (2.0**32 / b))][:32]
    assert len(boxes) == 32
    batch = pm.PMBatch(pm.make_config(np_side, n, 100.0, A_I, A_F, 4), boxes=boxes)
    batch.ic(list(range(32)))
    for r, box in enumerate(boxes):
        for mine, want in zip(batch.particles(r), _single(pm, np_side, n, box, r).particles()):
            assert torch.equal(mine, want), (r, box)


def test_launch_groups():
    pm = lib()
    np_side, n, nreal = 64, 64, 1026
    boxes = 200.0 + 3.0 * np.arange(nreal)
    batch = pm.PMBatch(pm.make_config(np_side, n, 1000.0, A_I, A_F, 4), boxes=boxes)
    batch.ic(list(range(nreal)))
    edges = np.array([1.0, 2.0, 4.0, 8.0, 16.0, 32.0])
    power = batch.power(edges)[1]
    for r in (0, 1, 127, 128, 255, 256, 1022, 1023, 1025):
        run = _single(pm, np_side, n, boxes[r], r)
        for mine, want in zip(batch.particles(r), run.particles()):
            assert torch.equal(mine, want), r
        np.testing.assert_allclose(power[r], run.power(edges)[1], rtol=1e-5)
