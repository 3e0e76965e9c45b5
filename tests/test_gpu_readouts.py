"""Nu / Sh and the residual where their launches change shape: one block and several per
wall, the most blocks (each thread then takes several positions), fewer blocks than the
residual's slots and many more; against the same numbers formed by numpy from the fields."""
import numpy as np
import pytest

from paper_1708_07525_gb300 import lbm

pytestmark = pytest.mark.gpu


def walls(c, T, w):
    """Mean wall gradients (Eq. 38) from a field T whose wall values are w."""
    n = c.nx if c.params.wall_lr == lbm.WALL_DIRICHLET else c.ny
    a = T if c.params.wall_lr == lbm.WALL_DIRICHLET else T.T
    s = -1.0 if c.params.wall_lr == lbm.WALL_DIRICHLET else 1.0
    d = (w[0] - w[1]) * (1.0 if s < 0 else -1.0)
    near = (-8.0 * w[0] + 9.0 * a[:, 0] - a[:, 1]) / 3.0
    far = -(-8.0 * w[1] + 9.0 * a[:, -1] - a[:, -2]) / 3.0
    return s * n * near.mean() / d, s * n * far.mean() / d


# 64 positions per block, 256 blocks per wall: 1 block, 2, ragged, the cap, beyond it
@pytest.mark.parametrize("nx,ny", [(3, 3), (5, 65), (64, 129), (9, 16384), (16500, 7), (7, 16500)])
@pytest.mark.parametrize("kind", ["cavity", "lid"])
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_wall_numbers_and_residual_match_the_fields(nx, ny, kind, precision):
    if kind == "cavity":
        p = lbm.lbm_derive_params(nx, ny, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0)
    else:
        p = lbm.lbm_derive_params_lid(nx, ny, 50.0, 1e3, 1e-2, 0.6, 1.0, 2.0, 1.0)
    c = lbm.Cavity(params=p, precision=precision, seed=5, noise=0.05)
    c.step(3)
    before = c.fields()
    assert c.residual() == np.inf
    c.step(2)
    now = c.fields()
    got = c.nusselt_sherwood() if kind == "cavity" else c.nusselt_sherwood_tb()
    again = c.nusselt_sherwood() if kind == "cavity" else c.nusselt_sherwood_tb()
    assert np.array_equal(got, again)        # fixed order, and the block count was put back
    w = (1.0, 0.0) if kind == "cavity" else (0.0, 1.0)
    (nl, nr), (sl, sr) = walls(c, now["T"], w), walls(c, now["C"], w)
    # the same FP64 arithmetic on the same values, in another order: n rounding errors of a
    # sum of n terms, and the FP32 reciprocals' (fields hold T0 + fl(sum / sigma) exactly)
    np.testing.assert_allclose(got, [nl, sl, nr, sr], rtol=1e-15 * (nx + ny), atol=1e-12)
    # differences are taken in the compute precision on T - T0: within two of its roundings
    u = 2.0 ** -52 if precision == "f64" else 2.0 ** -23
    r = max(np.abs(now[k] - before[k]).max() / np.abs(now[k]).max() for k in ("ux", "uy", "T", "C"))
    np.testing.assert_allclose(c.residual(), r, rtol=0, atol=4 * u)


@pytest.mark.parametrize("precision,layout,n", [("f32", "ab", 129), ("f32", "aa", 40), ("f64", "ab", 33),
                                                ("f32", "ab", 900)])
def test_a_few_steps_at_a_time(precision, layout, n):
    """A loop of short step calls, which replays captured chunks of eight steps after 64
    launches, takes the same steps as one call, from even and odd levels."""
    kw = dict(precision=precision, layout=layout, seed=2, noise=0.02)
    a = lbm.Cavity(n, n, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0, **kw)
    b = lbm.Cavity(n, n, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0, graph_chunk=-1, **kw)
    calls = [10, 9, 17, 8, 31, 1, 8, 16, 11, 24, 3, 40]
    for _ in range(2):
        for k in calls:
            a.step(k)
    b.step(2 * sum(calls))
    fa, fb = a.fields(), b.fields()
    for k in fa:
        assert np.array_equal(fa[k], fb[k]), k


def test_more_contexts_than_pinned_slots():
    """256 contexts read out through pinned memory, the others through copies; slots are
    taken again after contexts are gone."""
    made = [lbm.Cavity(8, 6, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0, precision="f32", seed=k) for k in range(262)]
    for c in made:
        c.step(2)
    got = [(tuple(c.nusselt_sherwood()), c.residual(), c.residual_parts()[4:].tolist()) for c in made]
    for c in made[:100]:
        c.close()
    for k in (0, 3, 255, 256, 261):
        c = lbm.Cavity(8, 6, 1e4, 1e-2, 0.6, 1.0, 2.0, 1.0, precision="f32", seed=k)
        c.step(2)
        assert (tuple(c.nusselt_sherwood()), c.residual(), c.residual_parts()[4:].tolist()) == got[k]
