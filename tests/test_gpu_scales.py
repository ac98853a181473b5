"""Length scales at which squares of coordinates leave single precision.

The list builders decide most pairs on FP32 offsets. On the FP32C path such a scale
has no meaning for the sums, but a list must hold nothing except particles. The FP64
path computes at every scale: a change of the unit of length by a power of two is
exact, so its lists stay the same.
"""
import numpy as np
import pytest

import paper_1904_00861_gb300 as dt

pytestmark = pytest.mark.gpu

F64, F32 = dt.DTSPH_FP64, dt.DTSPH_FP32C


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1904_00861_gb300 import build
    build.build()


def scattered(dim, ncell, n, scale, seed=3):
    """n particles at random in a periodic box of ncell cells a side, h = scale, a few of
    them in one cell and around it."""
    rng = np.random.default_rng(seed)
    L = 3.0 * (ncell + 0.5)
    x = rng.random((n, dim)) * L
    x[: n // 4] = x[0] + rng.random((n // 4, dim)) * 9.0 - 4.5
    x %= L
    cfg = dict(dim=dim, h=scale, m=scale ** dim, periodic=(1,) * dim + (0,) * (3 - dim), lo=(0.0,) * 3,
               hi=(L * scale,) * dim + (1.0,) * (3 - dim), nu=0.0, dt=0.01, max_neighbors=256)
    return cfg, x * scale


def lists(cfg, x, prec):
    sim = dt.Simulation(cfg, precision=prec, graph=1, lanes=4)
    sim.set_state(x, np.zeros_like(x), np.zeros(len(x)))
    dt.dtsph_build_neighbors(sim.ctx)
    out = [dt.dtsph_get_neighbors(sim.ctx, i) for i in range(len(x))]
    sim.close()
    return out


# 2D: 224 x 224 cells, 16,800 row segments (the builder of many segments); 3D
@pytest.mark.parametrize("dim,ncell,n", [(2, 224, 300), (3, 9, 200)])
def test_only_particles_are_listed_beyond_single_precision(dim, ncell, n):
    cfg, x = scattered(dim, ncell, n, 2.0 ** 70)
    for i, a in enumerate(lists(cfg, x, F32)):
        assert len(np.unique(a)) == len(a) and i not in a and (len(a) == 0 or (a.min() >= 0 and a.max() < n)), i


# the builder of few 2D cells, the one of many segments, 3D; (3h)^2 overflows FP32 from
# h = 2^62 on and is subnormal below h = 2^-64; at 2^61 an FP32 offset is finite still
@pytest.mark.parametrize("exponent", [-200, -80, -66, 61, 70, 200])
@pytest.mark.parametrize("dim,ncell,n", [(2, 12, 700), (2, 224, 300), (3, 9, 400)])
def test_fp64_lists_do_not_depend_on_the_unit_of_length(dim, ncell, n, exponent):
    cfg, x = scattered(dim, ncell, n, 1.0)
    want = lists(cfg, x, F64)
    assert max(len(a) for a in want) > 8
    cfg, x = scattered(dim, ncell, n, 2.0 ** exponent)
    for i, (a, b) in enumerate(zip(want, lists(cfg, x, F64))):
        assert np.array_equal(a, b), i
