"""The choice of the sort where some of the list shapes that commit times have more
cells than the one-cluster sort serves and others do not: it is timed when it serves the
default shape, a shape it does not serve takes the chain, and steps give the same bits
with either sort."""

import numpy as np
import pytest

from gpu_common import B, W, make

pytestmark = pytest.mark.gpu

MAX_CELLS = 1 << 20


def _cells(L, skin, m):
    return int(np.floor(L * m / ((1.58 + skin) * 1.0001))) ** 3


@pytest.mark.parametrize('L', [90.0, 92.0])
def test_sort_where_the_shapes_fall_on_both_sides_of_the_limit(L):
    bd = B()
    # 90: the default skin 0.2 fits, 0.15 does not; 92: 0.2 does not, 0.25 does
    assert (_cells(L, 0.2, 2) <= MAX_CELLS) == (L == 90.0)
    assert (_cells(L, 0.25, 2) <= MAX_CELLS) and _cells(L, 0.15, 2) > MAX_CELLS and _cells(L, 0.4, 3) > MAX_CELLS
    d = W.fluid_box(L=L, rho=0.004, n_species=1, seed=31)
    h = make(d)
    try:
        skin, m, tried = bd.tdpd_list_shape(h)
        sort, ms = bd.tdpd_sort_mode(h)
        lanes, mode = bd.tdpd_lanes(h), bd.tdpd_pair_mode(h)
        assert len(tried) == 10
        fits = _cells(L, np.float32(skin), m) <= MAX_CELLS
        assert (ms > 0).all() if L == 90.0 else (ms < 0).all(), (skin, m, sort, ms)
        assert (sort == 2) == (fits and L == 90.0 and ms[0] <= np.float32(1.03) * ms[1])
        assert L == 90.0 or (tried < 3 * tried.min()).all()      # (none with a sort that is not kept)
        bd.tdpd_step(h, 40)
        got = bd.tdpd_read_state(h, 0, 1) + bd.tdpd_read_forces(h, 0, 1)
    finally:
        bd.tdpd_destroy(h)
    g = bd.create_from(dict(d, lanes=lanes, pair_mode=mode, skin=skin, cells_per_cutoff=m))
    bd.tdpd_set_sort_mode(g, 2 if fits and sort == 1 else 1)
    try:
        bd.tdpd_step(g, 40)
        for x, y in zip(got, bd.tdpd_read_state(g, 0, 1) + bd.tdpd_read_forces(g, 0, 1)):
            assert np.array_equal(x, y)
    finally:
        bd.tdpd_destroy(g)
