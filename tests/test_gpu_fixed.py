"""The FP64 collision in block fixed point against the oracle where its scales are strained:
a state at rest, lattices of very different magnitudes, values far above and below one, a
node whose populations span many binades, rates at both ends of their range, and parameters
whose factors do not fit (which take the FP64 arithmetic)."""
import os

import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu


def rel(a, b):
    n = np.linalg.norm(b)
    return float(np.linalg.norm(a - b) / n) if n else float(np.abs(a).max())


# T and C deviate from T0 = C0 = 0 by these sizes, without buoyancy (the oracle holds absolute
# populations, whose rounding is more than a slow flow's; tests/test_gpu_parity.py has flows)
@pytest.mark.parametrize("ts,cs", [(0.0, 0.0), (1e-12, 1.0), (1e6, 1e-6)])
@pytest.mark.parametrize("layout", ["ab", "aa"])
@pytest.mark.parametrize("rate", [0.05, 1.95])
def test_scales_match_the_oracle(oracle_mod, ts, cs, layout, rate):
    oracle_mod.set_threads(os.cpu_count() or 1)
    nx, ny = 33, 18
    p = lbm.lbm_derive_params(nx, ny, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)
    o = oracle_mod.derive(nx, ny, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)
    rng = np.random.default_rng(3)
    # one node in ten carries 1e-9 of the others' deviation
    few = np.where(rng.uniform(size=(ny, nx)) < 0.1, 1e-9, 1.0)
    T, C = ts * few * rng.uniform(-1, 1, (ny, nx)), cs * rng.uniform(-1, 1, (ny, nx))
    for q in (p, o):
        q.T0 = q.C0 = 0.0
        for k in range(4):
            q.Tw[k], q.Cw[k] = (0.5 - k) * ts, (0.25 + k) * cs
        for k in (1, 2):
            q.zeta[k] = rate
        q.gbT = q.gbC = 0.0
    gpu = lbm.Cavity(params=p, precision="f64", layout=layout, T_init=T, C_init=C)
    ora = oracle_mod.Oracle(o, T_init=T, C_init=C)
    for n in (1, 2, 47):
        gpu.step(n)
        ora.step(n)
        fg, fo = gpu.fields(), ora.fields()
        # 50 steps of FP64 rounding on either side
        for k in ("T", "C"):
            assert rel(fg[k], fo[k]) <= 1e-13, (n, k)
        assert not fg["ux"].any() and not fg["uy"].any(), n


def test_factors_that_do_not_fit_take_fp64(oracle_mod):
    """sigma = 0.02 with varpi = 0.4: r_3 / 20 (4 - 5 varpi / sigma) = -7.2."""
    args = (24, 17, 1e3, 1e-2, 0.6, 1.0, 2.0, 1.0, 1.0, 0.02)
    p, o = lbm.lbm_derive_params(*args), oracle_mod.derive(*args)
    gpu = lbm.Cavity(params=p, precision="f64", seed=4, noise=0.01)
    ora = oracle_mod.Oracle(o, seed=4, noise=0.01)
    gpu.step(4)
    ora.step(4)
    for k in ("T", "C", "uy"):
        assert rel(gpu.fields()[k], ora.fields()[k]) <= 1e-12, k


def test_a_node_that_is_not_finite_is_found():
    T = np.full((20, 20), 0.5)
    T[7, 9] = np.inf
    c = lbm.Cavity(20, 20, 1e4, 1e-2, 0.6, 1.0, 1.0, 1.0, T_init=T, C_init=np.full((20, 20), 0.5))
    c.step(1)
    assert np.isnan(c.fields()["T"]).any()
    with pytest.raises(lbm.LbmError) as e:
        c.residual()
    assert e.value.status == lbm.ERR_DIVERGED
