"""When a step lets the next launch begin: at once, when the launch before it has completed, or
after its own end, by the blocks of its grid.  Every way keeps plain stream order (the bits
of ordinary launches), and no size takes much longer than a smaller one because waiting
launches fill the GPU."""
import time

import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu
LEGACY = 1          # cudaStreamLegacy: ordinary launches, no graphs


def cavity(precision, layout, walls, nx, ny, **kw):
    args = (nx, ny, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)
    if walls == "field":
        y, x = np.meshgrid((np.arange(ny) + 0.5) / ny, (np.arange(nx) + 0.5) / nx, indexing="ij")
        kw["eps_field"] = 0.6 * (1.0 + 0.1 * np.sin(2 * np.pi * x) * np.cos(np.pi * y))
    p = lbm.lbm_derive_params_nee(*args) if walls == "nee" else lbm.lbm_derive_params(*args)
    return lbm.Cavity(params=p, precision=precision, layout=layout, seed=3, noise=0.02, **kw)


# one block and several per SM; below, within and above each kernel's range
@pytest.mark.parametrize("precision,layout,walls", [
    ("f32", "ab", "halfway"), ("f32", "aa", "halfway"), ("f32", "ab", "nee"), ("f32", "ab", "field"),
    ("bf16", "ab", "halfway"), ("f16", "aa", "halfway"), ("f16", "aa", "field"), ("bf16", "ab", "nee"),
    ("f64", "ab", "halfway"), ("f64", "ab", "nee"), ("f64", "ab", "field"), ("f64", "aa", "halfway")])
@pytest.mark.parametrize("nx,ny", [(48, 48), (129, 128), (70, 300), (256, 240), (366, 366), (401, 300)])
def test_steps_keep_stream_order(precision, layout, walls, nx, ny):
    c, ref = cavity(precision, layout, walls, nx, ny), cavity(precision, layout, walls, nx, ny, stream=LEGACY)
    for n in (3, 64, 71):
        c.step(n)
        ref.step(n)
        a, b = (c.residual(), tuple(c.nusselt_sherwood())), (ref.residual(), tuple(ref.nusselt_sherwood()))
        assert a == b, n
    fc, fr = c.fields(), ref.fields()
    for k in fc:
        assert np.array_equal(fc[k], fr[k]), k


def step_time(*case):
    c = cavity(*case)
    c.step(256)
    times = []
    for _ in range(6):
        c.nusselt_sherwood()
        t0 = time.perf_counter()
        c.step(512)
        c.nusselt_sherwood()
        times.append(time.perf_counter() - t0)
    c.close()
    return min(times)


# 32 blocks on 32 SMs / 128 on 128 took 11.7 / 34 us; 711 / 744 of 760 places 4.9 / 13.4 us
@pytest.mark.parametrize("small,large", [
    (("f64", "ab", "field", 64, 64), ("f64", "ab", "field", 128, 128)),
    (("f64", "aa", "field", 64, 64), ("f64", "aa", "field", 128, 128)),
    (("bf16", "ab", "halfway", 352, 352), ("bf16", "ab", "halfway", 366, 366))])
def test_waiting_launches_do_not_crowd_a_step(small, large):
    assert step_time(*large) < 1.6 * step_time(*small)
