"""The pair kernel for more than two species and for the random flux (striped
lists), where it can go wrong: species counts around its compiled forms (odd ones
among them), several types, every lane width, particle counts that leave the last
warp and round partly empty, both shells, both list builds, batches, checkpoints of
both list layouts. Tolerances as in the per-step parity tests (gpu_common): the
sums are of the same terms."""

import struct

import numpy as np
import pytest

from gpu_common import B, W, check_step, forces_vs_oracle, make

pytestmark = pytest.mark.gpu


def _box(ns, seed, L=6.0, types=2, flux=False, reaction=True, rho=3.0, **kw):
    d = W.fluid_box(L=L, rho=rho, n_species=ns, seed=seed)
    rng = np.random.default_rng(seed)
    d['n_types'] = types
    for k in ('a', 'gamma', 'sigma'):
        d[k] = np.full((types, types), d[k][0, 0], np.float32)
    kap = rng.uniform(0.2, 2.0, (types, types, ns)).astype(np.float32)
    d['kappa'] = (0.5 * (kap + kap.transpose(1, 0, 2))).astype(np.float32)
    d['particles']['type'] = rng.integers(0, types, d['particles']['pos'].shape[0]).astype(np.int32)
    if reaction:
        d['reaction'] = dict(k=0.3, src=0, dst=ns - 1, types=1)
    if flux:
        d['random_flux'] = dict(m_s=0.05, rho=3.0)
    return dict(d, **kw)


@pytest.mark.parametrize('ns, types, flux, lanes, mode', [
    (3, 1, False, 1, 1), (3, 3, False, 2, 2), (4, 2, False, 32, 1), (5, 1, False, 8, 1), (9, 2, False, 16, 2),
    (10, 2, False, 4, 1), (10, 1, False, 32, 2), (11, 1, False, 8, 1), (16, 2, False, 4, 2), (16, 1, False, 1, 1),
    (2, 2, True, 8, 1), (3, 1, True, 4, 2), (10, 1, True, 16, 2), (16, 2, True, 2, 1)])
def test_forces_and_fluxes_match_oracle(ns, types, flux, lanes, mode):
    d = _box(ns, 500 + ns + lanes, types=types, flux=flux, lanes=lanes, pair_mode=mode)
    F, Q, Fo, Qo = forces_vs_oracle(d)
    check_step(F, Q, Fo, Qo, (ns, types, flux, lanes, mode))


@pytest.mark.parametrize('mode', [1, 2])
def test_dense_rows_match_oracle(mode):
    """Rows of more entries than a build thread keeps (8) until it may write them."""
    d = _box(3, 560, L=5.0, types=1, rho=16.0, lanes=4, pair_mode=mode)
    F, Q, Fo, Qo = forces_vs_oracle(d)
    check_step(F, Q, Fo, Qo, mode)


def _run(h, steps, ns, reps=1):
    bd = B()
    bd.tdpd_step(h, steps)
    bd.tdpd_sync(h)
    return [bd.tdpd_read_state(h, r, ns) + bd.tdpd_read_forces(h, r, ns) for r in range(reps)]


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize('ns, flux, mode', [(3, False, 1), (10, False, 2), (10, True, 2)])
def test_batch_equals_alone_over_rebuilds(ns, flux, mode):
    """Slots of a replica fall on other lanes, rounds and build threads in a batch
    (large enough for one build thread per particle) than alone: same bits."""
    bd = B()
    ds = [_box(ns, 600 + k, L=L, flux=flux, lanes=4, pair_mode=mode) for k, L in enumerate((5.1, 26.5, 6.3))]
    alone = []
    for d in ds:
        h = make(d)
        alone.append(_run(h, 12, ns)[0])
        assert bd.tdpd_list_rebuilds(h, 0) > 0
        bd.tdpd_destroy(h)
    hs = [bd.create_from(d) for d in ds]
    b = bd.tdpd_batch_create(hs)
    bd.tdpd_set_lanes(b, 4)
    bd.tdpd_set_pair_mode(b, mode)
    try:
        for k, got in enumerate(_run(b, 12, ns, 3)):
            assert _same(got, alone[k]), k
    finally:
        for h in hs + [b]:
            bd.tdpd_destroy(h)


def test_checkpoints_of_both_list_layouts(tmp_path):
    """A checkpoint continues with the same bits; a version 2 file (lists of one
    lane each, here left at zero) is accepted and its lists are rebuilt."""
    bd = B()
    ns, lanes = 3, 4
    d = _box(ns, 700, L=7.0, lanes=lanes, pair_mode=1)
    h = make(d)
    _run(h, 7, ns)
    path = str(tmp_path / 'c')
    bd.tdpd_save(h, path)
    want = _run(h, 9, ns)[0]
    bd.tdpd_load(h, path)
    assert _same(_run(h, 9, ns)[0], want)
    # the same state as a version 2 file: header fields, then the arrays in order
    raw = open(path, 'rb').read()
    size = struct.calcsize('<8sI11i')
    size += -size % 8 + 24
    head = list(struct.unpack_from('<8sI11i', raw))
    tail = struct.unpack_from('<qQQ', raw, size - 24)
    assert head[1] == 3
    N, lpp = head[2], head[7]
    nl, nlc = 4 * tail[2], 4 * N
    assert N == bd.tdpd_num_particles(h) and lpp == lanes
    body = raw[size:]
    xb = body[-(nl + 16 * N):-nl]
    front = body[:len(body) - nl - 16 * N - nlc]
    cap2 = 24
    ints = (N * lpp + 31) // 32 * 32 * cap2
    head[1], head[9] = 2, cap2
    pad = b'\0' * (size - 24 - struct.calcsize('<8sI11i'))
    old = (struct.pack('<8sI11i', *head) + pad + struct.pack('<qQQ', tail[0], tail[1], ints) + front +
           b'\0' * (4 * N * lpp) + xb + b'\0' * (4 * ints))
    open(path, 'wb').write(old)
    bd.tdpd_load(h, path)
    got = _run(h, 1, ns)[0]
    g = make(d)
    ref = _run(g, 8, ns)[0]
    bd.tdpd_destroy(g)
    bd.tdpd_destroy(h)
    # rebuilt lists change the order of the sums: equal to rounding
    for x, y in zip(got, ref):
        assert np.abs(x - y).max() <= 1e-5 * np.abs(y).max()
