"""A replica gives the same bits in a batch as alone (at equal lanes and pair mode)
when the other replicas of the batch differ in the number of types, in the random
flux or in the weight exponents, so that the batch takes other forms of the kernels
than the replica alone. Forces and fluxes of the forms that only the mixes reach
against the oracle, and checkpoints whose lists have the other layout."""

import struct

import numpy as np
import pytest

from gpu_common import B, W, check_step, forces_vs_oracle, make

pytestmark = pytest.mark.gpu

PLAIN, TYPES, FLUX, FLUX_TYPES, SOFT = dict(), dict(types=2), dict(flux=True), dict(types=2, flux=True), dict(s_f=0.41)


def _box(ns, seed, L, types=1, flux=False, s_f=2.0):
    d = W.fluid_box(L=L, rho=3.0, n_species=ns, seed=seed)
    rng = np.random.default_rng(seed)
    d['n_types'], d['s_f'] = types, s_f
    for k in ('a', 'gamma', 'sigma'):
        d[k] = np.full((types, types), d[k][0, 0], np.float32)
    kap = rng.uniform(0.2, 2.0, (types, types, ns)).astype(np.float32)
    d['kappa'] = (0.5 * (kap + kap.transpose(1, 0, 2))).astype(np.float32)
    d['particles']['type'] = rng.integers(0, types, d['particles']['pos'].shape[0]).astype(np.int32)
    if ns > 1:
        d['reaction'] = dict(k=0.3, src=0, dst=ns - 1, types=1)
    if flux:
        d['random_flux'] = dict(m_s=0.05, rho=3.0)
    return d


def _results(h, ns, replicas):
    bd = B()
    out = [[] for _ in range(replicas)]
    for steps in (0, 1, 11):                  # the loaded state, a step, rebuilds of the lists
        if steps:
            bd.tdpd_step(h, steps)
        bd.tdpd_sync(h)
        for r in range(replicas):
            out[r] += list(bd.tdpd_read_state(h, r, ns) + bd.tdpd_read_forces(h, r, ns))
    return out


@pytest.mark.parametrize('mix', [(PLAIN, TYPES), (PLAIN, FLUX), (TYPES, FLUX_TYPES), (FLUX, TYPES), (PLAIN, SOFT)])
@pytest.mark.parametrize('ns, lanes, mode', [(1, 1, 1), (1, 4, 2), (1, 32, 1), (2, 4, 1), (2, 1, 2), (2, 32, 2),
                                             (3, 4, 1), (3, 1, 2), (5, 4, 1), (8, 8, 2), (10, 1, 1), (10, 8, 1),
                                             (10, 8, 2), (16, 2, 1), (1, 2, 0), (2, 2, 0), (3, 8, 0)])
def test_batch_equals_alone_in_mixed_batches(mix, ns, lanes, mode):
    """mode 0: cell mode (skin 0)."""
    bd = B()
    skin, mode = (0.2, mode) if mode else (0.0, 1)
    ds = [dict(_box(ns, 50 + k + 7 * ns, 5.1 + k, **kw), lanes=lanes, pair_mode=mode, skin=skin)
          for k, kw in enumerate(mix)]
    alone = []
    for d in ds:
        h = make(d)
        alone.append(_results(h, ns, 1)[0])
        bd.tdpd_destroy(h)
    hs = [bd.create_from(d) for d in ds]
    b = bd.tdpd_batch_create(hs)
    for h in hs:
        bd.tdpd_destroy(h)
    try:
        bd.tdpd_set_lanes(b, lanes)
        bd.tdpd_set_pair_mode(b, mode)
        bd.tdpd_set_skin(b, skin)
        bd.tdpd_commit(b)
        for k, got in enumerate(_results(b, ns, len(ds))):
            for x, y in zip(got, alone[k]):
                assert np.array_equal(x, y), k
    finally:
        bd.tdpd_destroy(b)


@pytest.mark.parametrize('ns, types, lanes, mode', [(3, 2, 8, 1), (3, 1, 2, 2), (6, 1, 1, 1), (7, 2, 16, 2),
                                                    (8, 1, 4, 1), (8, 3, 32, 2), (9, 1, 4, 1), (9, 2, 1, 2)])
def test_forms_by_species_count_match_oracle(ns, types, lanes, mode):
    d = dict(_box(ns, 70 + ns + lanes, 6.0, types=types), lanes=lanes, pair_mode=mode)
    F, Q, Fo, Qo = forces_vs_oracle(d)
    check_step(F, Q, Fo, Qo, (ns, types, lanes, mode))


@pytest.mark.parametrize('ns, types, lanes, mode', [(1, 1, 1, 1), (1, 3, 4, 2), (1, 2, 32, 1), (2, 2, 2, 2),
                                                    (2, 1, 16, 1), (2, 3, 1, 2)])
def test_random_flux_of_few_species_matches_oracle(ns, types, lanes, mode):
    d = dict(_box(ns, 90 + ns + lanes, 6.0, types=types, flux=True), lanes=lanes, pair_mode=mode)
    F, Q, Fo, Qo = forces_vs_oracle(d)
    check_step(F, Q, Fo, Qo, (ns, types, lanes, mode))


def test_checkpoint_with_lists_per_particle_is_accepted(tmp_path):
    """A version 3 file (one list per particle, here left at zero) of a handle with two
    species and the random flux, whose lists are per lane: accepted, and the lists
    are rebuilt at the next step."""
    bd = B()
    ns, lanes = 2, 4
    d = dict(_box(ns, 96, 7.0, flux=True), lanes=lanes, pair_mode=1, skin=0.2)
    h = make(d)
    path = str(tmp_path / 'c')
    bd.tdpd_step(h, 7)
    bd.tdpd_save(h, path)
    raw = open(path, 'rb').read()
    size = struct.calcsize('<8sI11i')
    size += -size % 8 + 24
    head = list(struct.unpack_from('<8sI11i', raw))
    tail = struct.unpack_from('<qQQ', raw, size - 24)
    N, lpp = head[2], head[7]
    assert head[1] == 2 and N == bd.tdpd_num_particles(h) and lpp == lanes
    body, nl, nlc = raw[size:], 4 * tail[2], 4 * N * lanes
    xb = body[-(nl + 16 * N):-nl]
    front = body[:len(body) - nl - 16 * N - nlc]
    cap3 = 24
    ints = (N * lanes + 31) // 32 * 32 * (cap3 // lanes)
    head[1], head[9] = 3, cap3
    pad = b'\0' * (size - 24 - struct.calcsize('<8sI11i'))
    open(path, 'wb').write(struct.pack('<8sI11i', *head) + pad + struct.pack('<qQQ', tail[0], tail[1], ints) + front +
                           b'\0' * (4 * N) + xb + b'\0' * (4 * ints))
    want = _results(h, ns, 1)[0]
    bd.tdpd_load(h, path)
    got = _results(h, ns, 1)[0]
    bd.tdpd_destroy(h)
    # the same state; after a step its rebuilt lists change the order of the sums
    for k, (x, y) in enumerate(zip(got, want)):
        if k < 5:
            assert np.array_equal(x, y)
        elif k < 10:
            assert np.abs(x - y).max() <= 1e-5 * np.abs(y).max()
