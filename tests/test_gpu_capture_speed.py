"""A context whose steps have been captured by the caller keeps taking two steps per launch
(FP32, two buffers, 2048 x 2048: 1.45 times the time without), with the bits of single steps."""
import time

import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu
KEYS = ("ux", "uy", "T", "C")


def capture(c, st, n):
    import torch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        c.step(n)
    return g


# a caller captures fewer steps than graph_chunk (0: 64)
@pytest.mark.parametrize("before,n,graph_chunk", [(0, 2, 0), (2, 10, 0), (3, 12, 0), (6, 4, 0), (2, 10, -1),
                                                  (3, 4, 6), (0, 2, 6)])
def test_steps_after_a_capture_equal_single_steps(before, n, graph_chunk):
    import torch
    st = torch.cuda.Stream()
    args = (1000, 800, 1e5, 1e-2, 0.6, 1.0, 2.0, -1.0)
    a = lbm.Cavity(*args, precision="f32", seed=3, noise=0.02, stream=st.cuda_stream, graph_chunk=graph_chunk)
    b = lbm.Cavity(*args, precision="f32", seed=3, noise=0.02, block=(128, 1))
    a.step(before)
    g = capture(a, st, n)
    total = before
    for k in (2, 4, 7, 3, 66, 131):
        if total % 2 == before % 2:         # the parity it was captured at
            with torch.cuda.stream(st):
                g.replay()
            b.step(n)
        a.step(k)
        total += k
    b.step(total)
    fa, fb = a.fields(KEYS), b.fields(KEYS)
    for key in KEYS:
        assert np.array_equal(fa[key], fb[key]), key


def test_a_captured_context_keeps_its_speed():
    import torch

    def best(captured):
        st = torch.cuda.Stream()
        c = lbm.Cavity(2048, 2048, 1e5, 1e-3, 0.4, 1.0, 5.0, -1.0, precision="f32", stream=st.cuda_stream)
        if captured:
            capture(c, st, 4)
        c.step(64)
        times = []
        for _ in range(5):
            c.nusselt_sherwood()
            t0 = time.perf_counter()
            c.step(64)
            c.nusselt_sherwood()
            times.append(time.perf_counter() - t0)
        c.close()
        return min(times)

    assert best(True) < 1.2 * best(False)
