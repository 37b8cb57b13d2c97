"""A view that a caller holds across pm_batch_power stands where the batch does afterwards, as after
pm_batch_context, and measures the batch's current particles."""
import numpy as np
import pytest

from tests.gpu_util import lib

pytestmark = pytest.mark.gpu


def test_power_refreshes_held_views():
    pm = lib()
    cfg = pm.make_config(32, 64, 1000.0, 0.1, 1.0, 6)
    batch = pm.PMBatch(cfg, boxes=[1000.0, 2000.0])
    batch.ic([1, 2])
    view = batch.context(1)
    edges = np.array([1.0, 4.0, 16.0, 32.0])
    pm.pm_power(view, edges)
    assert pm.pm_state(view)[0] == 0
    for steps in (2, 4):
        batch.step(steps)
        power = batch.power(edges)[1]
        assert pm.pm_state(view) == batch.state()
        np.testing.assert_allclose(pm.pm_power(view, edges)[1], power[1], rtol=1e-5)
