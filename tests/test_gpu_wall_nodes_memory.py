"""Cavities with nodes on the walls take one step per launch and hold no second history for
two; a checkpoint that brings other walls still runs."""
import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu
ARGS = (1000, 800, 1e5, 1e-2, 0.6, 1.0, 2.0, -1.0)


def test_wall_nodes_hold_no_second_history():
    nodes = lbm.Cavity(params=lbm.lbm_derive_params_nee(*ARGS), precision="f32", seed=3, noise=0.02)
    tiled = lbm.Cavity(params=lbm.lbm_derive_params_nee(*ARGS), precision="f32", block=(128, 1))
    halfway = lbm.Cavity(*ARGS, precision="f32", seed=4, noise=0.02)
    assert nodes.steps_per_launch() == 1 and halfway.steps_per_launch() == 2
    assert nodes.device_bytes() == tiled.device_bytes()
    assert halfway.device_bytes() - nodes.device_bytes() == 16 * 800 * 1024
    # each takes the other's walls with its state
    halfway.step(6), nodes.step(6)
    mine, other = halfway.save(), nodes.save()
    halfway.load(other), nodes.load(mine)
    assert (nodes.steps_per_launch(), halfway.steps_per_launch()) == (1, 1)
    tiled.load(other)
    for c in (halfway, tiled):
        c.step(5)
    plain = lbm.Cavity(*ARGS, precision="f32", block=(128, 1))
    plain.load(mine)
    for c in (nodes, plain):
        c.step(5)
    for a, b in ((halfway, tiled), (nodes, plain)):
        fa, fb = a.fields(), b.fields()
        for k in fa:
            assert np.array_equal(fa[k], fb[k]), k
