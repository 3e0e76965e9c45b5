"""Steps captured by the caller: an even number of them can be replayed, also with other
steps in between, whatever launches the context would take by itself."""
import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,precision,layout,before", [
    (1000, 800, "f32", "ab", 65), (1000, 800, "f32", "ab", 6), (96, 64, "f32", "ab", 70), (96, 64, "f64", "ab", 70),
    (96, 64, "f32", "aa", 70), (96, 64, "f64", "aa", 6)])
def test_captured_steps_can_be_replayed(nx, ny, precision, layout, before):
    import torch
    st = torch.cuda.Stream()
    args = (nx, ny, 1e5, 1e-2, 0.6, 1.0, 2.0, -1.0)
    a = lbm.Cavity(*args, precision=precision, layout=layout, seed=3, noise=0.02, stream=st.cuda_stream)
    b = lbm.Cavity(*args, precision=precision, layout=layout, seed=3, noise=0.02)
    for _ in range(before - 2):
        a.step(1)                             # single launches, then two steps at once
    a.step(2)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.step(10)
    with torch.cuda.stream(st):
        g.replay()
        g.replay()
    a.step(4)
    a.step(64)
    with torch.cuda.stream(st):
        g.replay()
    b.step(before + 30 + 68)
    fa, fb = a.fields(), b.fields()
    for k in ("ux", "uy", "T", "C"):
        assert np.array_equal(fa[k], fb[k]), k
