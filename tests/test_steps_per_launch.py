"""How many time steps a launch takes, as the library reports it and as the benchmark counts
its launches by it."""
import pytest

import bench
from paper_1708_07525_gb300 import lbm


def test_launches_of_the_benchmark():
    assert [bench.step_launches(p, k) for p, k in ((1, 100), (1, 1), (2, 100), (2, 101), (2, 1))] == [100, 1, 50, 51, 1]


def test_no_context_takes_no_steps():
    assert lbm.lib().lbm_steps_per_launch(None) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,two", [
    (1000, 750, True), (1000, 749, False),
    (7328, 7300, True), (7328, 7360, False),     # byte offsets of a state plane set beyond 32 bits
])
def test_steps_per_launch_of_a_cavity(nx, ny, two):
    args = (nx, ny, 1e5, 1e-2, 0.6, 1.0, 2.0, -1.0)
    with lbm.Cavity(*args, precision="f32") as c:
        assert c.steps_per_launch() == (2 if two else 1)
    for kw in (dict(block=(128, 1)), dict(layout="aa"), dict(precision="bf16")):
        with lbm.Cavity(*args, **{"precision": "f32", **kw}) as c:
            assert c.steps_per_launch() == 1, kw
