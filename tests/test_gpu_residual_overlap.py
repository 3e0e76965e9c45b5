"""lbm_residual_noalloc of several contexts at once, each on its own stream and host thread:
the numbers of one context at a time."""
import threading

import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu
CASES = [(700, 900, "f32"), (1024, 512, "f32"), (301, 257, "f64"), (640, 640, "bf16")]


def run(case, seed):
    import torch
    nx, ny, precision = case
    c = lbm.Cavity(nx, ny, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0, precision=precision, seed=seed, noise=0.02)
    snap = torch.zeros(4 * nx * ny, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    got = []
    for k in range(150):
        c.step(2)
        got.append(c.residual_noalloc(snap.data_ptr(), k > 0))
    return got


def test_overlapping_calls_give_the_numbers_of_single_ones():
    alone = [run(case, k) for k, case in enumerate(CASES)]
    together = [None] * len(CASES)

    def go(k):
        together[k] = run(CASES[k], k)

    threads = [threading.Thread(target=go, args=(k,)) for k in range(len(CASES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert together == alone
