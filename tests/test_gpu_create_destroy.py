"""A program with one cavity at a time: making one and closing it costs little more than
beside others, and its read-outs are right each time."""
import gc
import time

import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu
ARGS = (64, 64, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)


def test_a_lone_cavity_is_made_and_closed_as_quickly_as_one_beside_others():
    gc.collect()                                  # no cavity of another test is left

    def typical(read):
        times, got = [], set()
        for _ in range(25):
            t0 = time.perf_counter()
            c = lbm.Cavity(*ARGS, precision="f32", seed=3, noise=0.02)
            if read:
                c.step(4)
                got.add((tuple(c.nusselt_sherwood()), c.residual(), tuple(c.residual_parts())))
            c.close()
            times.append(time.perf_counter() - t0)
        assert len(got) == (1 if read else 0)
        return sorted(times)[12]

    alone = typical(False), typical(True)
    other = lbm.Cavity(*ARGS, precision="f32")
    beside = typical(False), typical(True)
    other.close()
    assert alone[0] < 3 * beside[0] and alone[1] < 3 * beside[1], (alone, beside)
