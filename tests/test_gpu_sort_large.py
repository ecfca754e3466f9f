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


def test_reload_of_a_sparse_box_gives_the_same_bits():
    """Far more cells than particles: the counters a load clears are not covered
    by a thread per particle."""
    bd = B()
    d = W.fluid_box(L=90.0, rho=0.0004, n_species=1, seed=8)
    p = d['particles']
    n = p['pos'].shape[0]
    assert 100 < n < 600
    p['pos'][1] = p['pos'][0]
    p['pos'][1, 0] += np.float32(0.4) if p['pos'][0, 0] < 80 else np.float32(-0.4)
    # two handles with different histories of the same length (the step number keys
    # the random force), then the same state
    got = []
    for shift in (0.0, 7.0):
        q = dict(p, pos=np.mod(p['pos'] + np.float32(shift), np.float32(90.0)).astype(np.float32) % np.float32(90.0))
        h = make(dict(d, particles=q, lanes=4, skin=0.15))
        try:
            bd.tdpd_step(h, 20)
            bd.tdpd_set_state(h, 0, p['pos'], p['vel'], p['conc'])
            loaded = bd.tdpd_read_forces(h, 0, 1)
            bd.tdpd_step(h, 20)
            got.append(loaded + bd.tdpd_read_state(h, 0, 1))
        finally:
            bd.tdpd_destroy(h)
    assert np.abs(got[0][0][:2]).max() > 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)
