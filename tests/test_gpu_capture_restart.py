"""Steps captured by the caller, replayed after a reset or a load: the replay takes the new
run's steps, whatever buffers the context was on when the steps were captured and however
many steps it took since (1000 x 800 in FP32 takes two steps per launch)."""
import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu
KEYS = ("ux", "uy", "T", "C")


def cavity(precision, layout, seed, stream=None):
    nx, ny = (1000, 800) if precision == "f32" and layout == "ab" else (96, 64)
    return lbm.Cavity(nx, ny, 1e5, 1e-2, 0.6, 1.0, 2.0, -1.0, precision=precision, layout=layout, seed=seed,
                      noise=0.02, stream=stream)


# steps before the capture (an even level: no swap, one, two, 32 and one), steps after it
@pytest.mark.parametrize("before,after", [(0, 0), (2, 0), (2, 1), (4, 3), (6, 2), (66, 65)])
@pytest.mark.parametrize("how", ["reset", "load"])
@pytest.mark.parametrize("precision,layout", [("f32", "ab"), ("f64", "ab"), ("f32", "aa")])
def test_replay_after_a_new_state(precision, layout, how, before, after):
    import torch
    st = torch.cuda.Stream()
    a, b = cavity(precision, layout, 3, st.cuda_stream), cavity(precision, layout, 9)
    a.step(before)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.step(10)
    a.step(after)
    for _ in range(2):
        if how == "reset":
            a.reset(seed=9, noise=0.02)
            b.reset(seed=9, noise=0.02)
        else:
            b.step(4)
            a.load(b.save())
        assert a.t == b.t
        with torch.cuda.stream(st):
            g.replay()
        a.step(3)
        b.step(13)
        fa, fb = a.fields(KEYS), b.fields(KEYS)
        for k in KEYS:
            assert np.array_equal(fa[k], fb[k]), k
        b.step(1)
        a.step(1)


def test_a_captured_reset_restarts_the_run():
    """The reset is in the caller's graph, alone; the context then takes steps by itself."""
    import torch
    st = torch.cuda.Stream()
    a, b = cavity("f32", "ab", 3, st.cuda_stream), cavity("f32", "ab", 9)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.reset(seed=9, noise=0.02)
    a.step(2)
    with torch.cuda.stream(st):
        g.replay()
    fa, fb = a.fields(KEYS), b.fields(KEYS)
    for k in KEYS:
        assert np.array_equal(fa[k], fb[k]), k
