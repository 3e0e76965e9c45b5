"""In-place cavities whose odd step has its ring in the same launch: even steps whose grid all but
fills the GPU (1,200 blocks of 1,216 that fit) take no longer than slightly smaller ones, and
keep plain stream order.  The same for 16-bit steps with nodes on the walls, two of whose
grids fill it."""
import numpy as np
import pytest

from test_gpu_step_start import LEGACY, cavity, step_time

pytestmark = pytest.mark.gpu


# 5.9 / 12.3, 5.4 / 10.5 and 7.8 / 12.2 us per step when the next launch is let in at once
@pytest.mark.parametrize("small,large", [
    (("f16", "aa", "halfway", 501, 290), ("f16", "aa", "halfway", 501, 301)),
    (("f32", "aa", "halfway", 363, 390), ("f32", "aa", "halfway", 383, 402)),
    (("bf16", "ab", "nee", 140, 285), ("bf16", "ab", "nee", 140, 300))])
def test_a_grid_that_fills_the_gpu_is_not_crowded(small, large):
    assert step_time(*large) < 1.4 * step_time(*small)


@pytest.mark.parametrize("case", [
    ("f32", "aa", "halfway", 501, 301), ("f32", "aa", "field", 501, 301), ("f16", "aa", "halfway", 501, 301),
    ("f16", "aa", "field", 501, 301), ("bf16", "ab", "nee", 140, 300)])
def test_steps_keep_stream_order(case):
    c, ref = (cavity(*case, **kw) for kw in ({}, {"stream": LEGACY}))
    for n in (3, 64, 71):
        c.step(n)
        ref.step(n)
        assert (c.residual(), tuple(c.nusselt_sherwood())) == (ref.residual(), tuple(ref.nusselt_sherwood())), n
    fc, fr = c.fields(), ref.fields()
    for k in fc:
        assert np.array_equal(fc[k], fr[k]), k
