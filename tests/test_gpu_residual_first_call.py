"""A first residual that is refused, because the stream is being captured, leaves nothing behind
that later ones would trip over.  The device memory comes from a pool that holds other
values, as reused memory does."""
import ctypes as C

import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu


class Pool:
    """Allocator hooks that hand out pieces of one block of bytes 0xFF."""

    def __init__(self):
        import torch
        self.block = torch.full((16 << 20,), 255, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        self.at = 0

        def take(nbytes, user, stream):
            p = self.block.data_ptr() + self.at
            self.at += -(-int(nbytes) // 256) * 256
            return p if self.at <= self.block.numel() else None

        self.alloc, self.free = lbm.ALLOC_FN(take), lbm.FREE_FN(lambda p, user, stream: None)


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_residual_after_one_in_a_capture(precision, monkeypatch):
    import torch
    st = torch.cuda.Stream()
    kw = dict(precision=precision, seed=3, noise=0.02)
    args = (64, 48, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)
    b = lbm.Cavity(*args, **kw)
    monkeypatch.setattr(lbm, "TorchAllocator", Pool)
    a = lbm.Cavity(*args, stream=st.cuda_stream, **kw)
    a.step(5), b.step(5)
    torch.cuda.synchronize()
    cuda, graph = C.CDLL("libcuda.so.1"), C.c_void_p()
    assert cuda.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 2) == 0
    with pytest.raises(lbm.LbmError):
        a.residual()
    assert cuda.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(graph)) != 0
    for _ in range(2):                        # the refusal may be reported once more
        try:
            a.residual()
        except lbm.LbmError:
            pass
    b.residual()
    for _ in range(2):
        a.step(7), b.step(7)
        assert a.residual() == b.residual() > 0
        assert np.array_equal(a.residual_parts(), b.residual_parts())
