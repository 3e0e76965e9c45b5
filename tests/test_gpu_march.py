"""Two steps per launch (FP32, two buffers, from 750,000 nodes on) against one step per
launch: the same bits, over ragged strips and bands, odd numbers of steps, moving walls,
graph replay from every pair of buffers, and a checkpoint in between."""
import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu
KEYS = ("ux", "uy", "T", "C", "rho")


def params(nx, ny, lid):
    if lid:
        return lbm.lbm_derive_params_lid(nx, ny, 100.0, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)
    return lbm.lbm_derive_params(nx, ny, 1e5, 1e-2, 0.6, 1.0, 2.0, -1.0)


# strips of 24 columns: exact, one column over, one short; bands of 4 to 32 rows: ragged, odd;
# fewer rows than a band; a single strip
@pytest.mark.parametrize("nx,ny", [(1008, 745), (889, 845), (863, 870), (250003, 3), (13, 57700)])
@pytest.mark.parametrize("lid", [False, True], ids=["cavity", "lid"])
def test_two_steps_per_launch_equal_single_steps(nx, ny, lid):
    p = params(nx, ny, lid)
    a = lbm.Cavity(params=p, precision="f32", seed=3, noise=0.02)
    b = lbm.Cavity(params=p, precision="f32", seed=3, noise=0.02)
    for n in (2, 5, 64, 1, 66):              # 64 and 66 replay graphs from different buffers
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert a.t == b.t
    fa, fb = a.fields(), b.fields()
    for k in KEYS:
        assert np.array_equal(fa[k], fb[k]), k
    a.residual(), b.residual()
    blob = a.save()
    a.step(7)
    again = a.fields()
    a.load(blob)
    a.step(4)
    a.step(3)
    b.step(1), b.step(6)
    for k in KEYS:
        assert np.array_equal(a.fields()[k], again[k]) and np.array_equal(b.fields()[k], again[k]), k
    assert a.residual() == np.inf            # a loaded state has no earlier fields
