"""The membrane kernel over its range of meshes and cluster sizes: the smallest and
the largest mesh against the oracle (per-step tolerances of gpu_common), and the
same bits alone (four CTAs per membrane) and in batches of many membranes (two CTAs,
one CTA), lagged constraints included."""

import numpy as np
import pytest

from gpu_common import B, W, check_step, forces_vs_oracle, make

pytestmark = pytest.mark.gpu


def _cell(nv, seed, L=9.0, lagged=0):
    """A perturbed spherical cell of nv vertices across a periodic corner."""
    d = W.single_rbc(L=L, nv=500, diameter=5.0, seed=seed)
    rng = np.random.default_rng(seed)
    verts, tri = W.sphere_mesh(nv, 2.2)
    d['rbcs'] = [W.place_rbc(verts, tri, (0.3, L - 0.2, 0.5 * L), d['L'], rng)]
    d['membrane']['lagged_av'] = lagged
    return W.perturb(d, seed + 1, dx=0.02 * 2.2 / np.sqrt(nv / 12.0), rbc_scale=1.02)


@pytest.mark.parametrize('nv', [4, 12, 63, 512, 1024])
def test_mesh_sizes_match_oracle(nv):
    d = _cell(nv, 800 + nv)
    F, Q, Fo, Qo = forces_vs_oracle(d)
    check_step(F, Q, Fo, Qo, nv)


@pytest.mark.parametrize('replicas, lagged', [(2, 0), (80, 0), (160, 0), (160, 1)])
def test_same_bits_for_every_cluster_size(replicas, lagged):
    bd = B()
    ds = [dict(_cell((63, 500, 12)[k % 3], 900 + k, lagged=lagged), lanes=1, pair_mode=2) for k in range(replicas)]
    hs = [bd.create_from(d) for d in ds]
    b = bd.tdpd_batch_create(hs)
    for h in hs:
        bd.tdpd_destroy(h)
    bd.tdpd_set_lanes(b, 1)
    bd.tdpd_set_pair_mode(b, 2)
    try:
        bd.tdpd_step(b, 3)
        bd.tdpd_sync(b)
        for k in (0, 1, replicas - 1):
            h = make(ds[k])
            bd.tdpd_step(h, 3)
            bd.tdpd_sync(h)
            for x, y in zip(bd.tdpd_read_state(b, k, 1) + bd.tdpd_read_forces(b, k, 1) + bd.tdpd_read_rbc(b, k, 1),
                            bd.tdpd_read_state(h, 0, 1) + bd.tdpd_read_forces(h, 0, 1) + bd.tdpd_read_rbc(h, 0, 1)):
                assert np.array_equal(x, y), k
            bd.tdpd_destroy(h)
    finally:
        bd.tdpd_destroy(b)
