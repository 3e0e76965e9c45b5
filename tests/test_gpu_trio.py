"""Three warps for 32 nodes (FP64, two buffers, small cavities) against the cavity in two slabs,
which has one thread a node (the same bits), and, with nodes on the walls, against the
oracle: sizes about a multiple of 32 nodes and on both sides of the largest."""
import os

import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm
from test_gpu_slab import exchange

pytestmark = pytest.mark.gpu
KEYS = ("ux", "uy", "T", "C")


@pytest.mark.parametrize("nx,ny", [(3, 3), (8, 4), (3, 11), (31, 33), (3, 20833), (250, 250), (251, 250)])
@pytest.mark.parametrize("lid", [False, True], ids=["cavity", "lid"])
def test_halfway_walls_equal_slabs(nx, ny, lid):
    import torch
    p = (lbm.lbm_derive_params_lid(nx, ny, 100.0, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0) if lid else
         lbm.lbm_derive_params(nx, ny, 1e4, 1e-2, 0.6, 1.0, 2.0, -1.0))
    whole = lbm.Cavity(params=p, precision="f64", seed=3, noise=0.02)
    cut = ny // 2
    slabs = [lbm.Cavity(params=p, slab=s, precision="f64", seed=3, noise=0.02) for s in ((0, cut), (cut, ny - cut))]
    faces = [[torch.empty(slabs[0].halo_bytes(), dtype=torch.uint8, device="cuda") for _ in range(2)] for _ in slabs]
    for n in (1, 2, 65):
        whole.step(n)
        for _ in range(n):
            for s in slabs:
                s.step(1)
            exchange(slabs, faces)
        fw, fs = whole.fields(), [s.fields() for s in slabs]
        for k in KEYS:
            assert np.array_equal(np.concatenate([f[k] for f in fs]), fw[k]), (n, k)


@pytest.mark.parametrize("nx,ny,steps", [(5, 5, 60), (18, 18, 60), (10, 23, 60), (300, 300, 3), (301, 300, 3)])
def test_wall_nodes_match_the_oracle(oracle_mod, nx, ny, steps):
    oracle_mod.set_threads(os.cpu_count() or 1)
    args = (nx, ny, 1e4, 1e-2, 0.6, 1.0, 3.0, -1.5)
    p, o = lbm.lbm_derive_params_nee(*args), oracle_mod.derive(*args, nee=True)
    for q in (p, o):
        q.uw[3][0] = 0.05
        q.BiC[1] = 7.0
    gpu = lbm.Cavity(params=p, precision="f64", seed=5, noise=0.02)
    ora = oracle_mod.Oracle(o, seed=5, noise=0.02)
    gpu.step(steps)
    ora.step(steps)
    fg, fo = gpu.fields(), ora.fields()
    for f in (fg, fo):
        f["u"] = np.stack([f["ux"], f["uy"]])
    for k in ("u", "T", "C"):                 # at most 60 steps of FP64 rounding on either side
        assert np.linalg.norm(fg[k] - fo[k]) <= 1e-12 * np.linalg.norm(fo[k]), k


def test_a_node_that_is_not_finite_is_found_with_wall_nodes():
    T = np.full((20, 20), 0.5)
    T[7, 9] = np.inf
    c = lbm.Cavity(params=lbm.lbm_derive_params_nee(20, 20, 1e4, 1e-2, 0.6, 1.0, 1.0, 1.0), T_init=T,
                   C_init=np.full((20, 20), 0.5))
    c.step(1)
    assert np.isnan(c.fields()["T"]).any()
    with pytest.raises(lbm.LbmError) as e:
        c.residual()
    assert e.value.status == lbm.ERR_DIVERGED
