"""The sort of a rebuild step where a CTA of the binning takes several turns: a
system above what one turn of its grid covers, alone and in a batch large enough
that the decision is taken by its own kernel and the grid is not limited. A
replica's bits are the same alone and in a batch."""

import numpy as np
import pytest

from gpu_common import B, W, make

pytestmark = pytest.mark.gpu


def _state(h, ns):
    bd = B()
    bd.tdpd_step(h, 12)
    bd.tdpd_sync(h)
    assert bd.tdpd_list_rebuilds(h, 0) >= 2
    return bd.tdpd_read_state(h, 0, ns) + bd.tdpd_read_forces(h, 0, ns)


def test_binning_turns_give_the_same_bits():
    bd = B()
    kw = dict(lanes=1, pair_mode=2, skin=0.15)
    big = dict(W.fluid_box(L=60.0, rho=3.0, n_species=1, seed=5), **kw)
    assert big['particles']['pos'].shape[0] > 2 * 256 * 152 * 8
    small = [dict(W.fluid_box(L=5.1, rho=3.0, n_species=1, seed=6 + k), **kw) for k in range(17)]
    h = make(big)
    alone = _state(h, 1)
    bd.tdpd_destroy(h)
    hs = [bd.create_from(d) for d in [big] + small]
    h = bd.tdpd_batch_create(hs)
    for x in hs:
        bd.tdpd_destroy(x)
    bd.tdpd_set_lanes(h, 1)
    bd.tdpd_set_pair_mode(h, 2)
    bd.tdpd_set_skin(h, 0.15)
    bd.tdpd_commit(h)
    both = _state(h, 1)
    bd.tdpd_destroy(h)
    for a, b in zip(alone, both):
        assert np.array_equal(a, b)
