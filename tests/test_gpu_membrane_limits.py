"""The membrane kernel's splits over CTAs and threads, up to the limit of its shared
memory (one CTA for a mesh of 1024 vertices), and handles of different meshes committed
by several threads at once."""

import threading

import numpy as np
import pytest

from gpu_common import B, W, make

pytestmark = pytest.mark.gpu


def _cell(nv, seed, L=9.0):
    d = W.single_rbc(L=L, nv=500, diameter=5.0, seed=seed)
    rng = np.random.default_rng(seed)
    verts, tri = W.sphere_mesh(nv, 2.2)
    d['rbcs'] = [W.place_rbc(verts, tri, (0.3, L - 0.2, 0.5 * L), d['L'], rng)]
    d = W.perturb(d, seed + 1, dx=0.02 * 2.2 / np.sqrt(nv / 12.0), rbc_scale=1.02)
    return dict(d, lanes=1, pair_mode=2, skin=0.2)


def _run(h, replica):
    bd = B()
    return bd.tdpd_read_state(h, replica, 1) + bd.tdpd_read_forces(h, replica, 1) + bd.tdpd_read_rbc(h, replica, 1)


@pytest.mark.parametrize('mode', [1, 2])
@pytest.mark.parametrize('lagged', [0, 1])
@pytest.mark.parametrize('sizes, replicas', [((1024,), 100), ((1024, 600), 153), ((4, 66, 12), 153), ((4, 67, 12), 153),
                                             ((500, 63), 17), ((4, 1024), 37), ((500, 162), 77), ((513, 4), 16)])
def test_same_bits_for_every_split(sizes, replicas, lagged, mode):
    """Up to 16 membranes take eight CTAs of 512 threads each, of 256 beside the half
    shell's walk for at most 512 vertices; 17 take four, 37 two, 77 and 100 one, 153 two
    of the largest meshes, one of the smaller, and of the smallest one with 128
    threads: the same bits alone and in a batch, over steps that pass totals on to the
    next (a lagged membrane's are added by one CTA of the cluster)."""
    bd = B()
    ds = [dict(_cell(sizes[k % len(sizes)], 950 + k % 6), pair_mode=mode) for k in range(replicas)]
    for d in ds:
        d['membrane'] = dict(d['membrane'], lagged_av=lagged)
    hs = [bd.create_from(d) for d in ds]
    b = bd.tdpd_batch_create(hs)
    for h in hs:
        bd.tdpd_destroy(h)
    bd.tdpd_set_lanes(b, 1)
    bd.tdpd_set_pair_mode(b, mode)
    bd.tdpd_set_skin(b, 0.2)
    try:
        bd.tdpd_step(b, 3)
        bd.tdpd_sync(b)
        for k in (0, 1, 2, replicas - 1):
            h = make(ds[k])
            bd.tdpd_step(h, 3)
            bd.tdpd_sync(h)
            for x, y in zip(_run(b, k), _run(h, 0)):
                assert np.array_equal(x, y), k
            bd.tdpd_destroy(h)
    finally:
        bd.tdpd_destroy(b)


def test_threads_commit_different_meshes():
    """Both meshes need more shared memory than a launch has by default."""
    bd = B()
    want, done = {}, []
    ds = {nv: _cell(nv, 960) for nv in (700, 1024)}

    def run(nv):
        h = make(ds[nv])
        bd.tdpd_step(h, 2)
        bd.tdpd_sync(h)
        out = _run(h, 0)
        bd.tdpd_destroy(h)
        return out

    def work(nv):
        for _ in range(8):
            done.append(all(np.array_equal(x, y) for x, y in zip(run(nv), want[nv])))

    for nv in ds:
        want[nv] = run(nv)
    threads = [threading.Thread(target=work, args=(nv,)) for nv in list(ds) * 2]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(done) == 32 and all(done)
