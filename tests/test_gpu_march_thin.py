"""Thin cavities of 750,000 nodes and more: two steps per launch only where strips and bands
repeat little of the work, and there with the bits of one step per launch."""
import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,two", [
    (250000, 3, False), (187500, 4, False), (150000, 5, False), (125000, 6, True), (107143, 7, False),
    (93750, 8, True), (83334, 9, True), (31, 24194, True), (32, 23438, False), (33, 22728, True)])
def test_thin_cavities(nx, ny, two):
    args = (nx, ny, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)
    a = lbm.Cavity(*args, precision="f32", seed=3, noise=0.02)
    b = lbm.Cavity(*args, precision="f32", seed=3, noise=0.02, block=(32, 4))
    assert (a.steps_per_launch(), b.steps_per_launch()) == (2 if two else 1, 1)
    # no second history where a launch takes one step (16 bytes per node of a padded row)
    more = 16 * ny * -(-nx // 32) * 32 if two else 0
    assert a.device_bytes() - b.device_bytes() == more
    a.step(7)
    b.step(7)
    fa, fb = a.fields(), b.fields()
    for k in fa:
        assert np.array_equal(fa[k], fb[k]), k
