"""Timed cases of the tDPD + RBC framework: what a user's program asks of it,
through the C ABI's Python binding, from a 4000-particle box to batches of
close to a million particles, and the surrogate network's calls.

A case is a dict of plain values. ``prepare`` builds what the program holds
before the call (a committed handle and the buffers its results go to, or
the inputs of a call that takes arrays), ``run`` makes the call once, and
``exact`` gives the same outputs in binary64 from plain torch.

Kinds:
  step     a running simulation advanced by ``steps`` time steps, then its
           state read into device memory (the loop of every simulation: run
           to the next output, read, go on)
  reload   a state from pinned host memory loaded into a committed handle,
           one step, state and observables read back (a sweep or an outer
           solver that owns the state)
  forces   the allocation-free pair force and flux of device arrays
  train    Adam steps of the surrogate ensemble, loss and parameters back
  predict  the surrogate ensemble's prediction for new parameter points
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

import workloads as W
from workloads import surrogate as WS
from paper_1611_06163_gb300 import binding as bd


def listed():
    return [
        # the plain tDPD fluid of the quick checks: 4000 particles, where the
        # launches and the latency of each kernel are everything
        dict(name='fluid_4k', kind='step', system='fluid', L=10.0, rho=4.0, species=1, steps=8),
        # one red cell in solvent, the paper's unit system (24,500 particles)
        dict(name='single_rbc', kind='step', system='rbc', L=20.0, diameter=8.0, steps=8),
        # the cell suspension between walls: 40 cells, two species, a
        # reaction, frozen wall particles (255,000 particles with the walls)
        dict(name='channel', kind='step', system='channel', L=64.0, W=32.0, H=32.0, cells=40, steps=4),
        # a parameter sweep's batch of uneven replicas (841,000 particles)
        dict(name='ensemble_128', kind='step', system='ensemble', replicas=128, steps=8),
        # a plain fluid that exceeds the L2 cache, one species
        dict(name='fluid_786k', kind='step', system='fluid', L=64.0, rho=3.0, species=1, steps=4),
        # the paper's ten-species fluid, a box of ragged size
        dict(name='fluid_10_species', kind='step', system='fluid', L=45.7, rho=3.0, species=10, steps=4),
        # the flow validation: weight exponent 0.41 and the long force cut-off
        # (256,000 particles, every pair inside r_cc has a force)
        dict(name='poiseuille', kind='step', system='poiseuille', L=40.0, rho=4.0, species=1, steps=1),
        # the random flux of Eq. 7 on ten species, the transport option whose
        # every pair draws random numbers (41,000 particles)
        dict(name='random_flux', kind='step', system='random_flux', L=24.0, rho=3.0, species=10, steps=2),
        # a state owned by the host loaded, stepped once and read back
        dict(name='reload_rbc', kind='reload', system='rbc', L=20.0, diameter=8.0, steps=1),
        # pair forces inside another engine's step, its own device arrays
        dict(name='forces_12k', kind='forces', system='fluid', L=15.9, rho=3.0, species=2, steps=1),
        # the surrogate's training at its configured size
        dict(name='train_4096', kind='train', members=5, samples=4096, steps=2),
        # ranking a sweep's candidates with the ensemble
        dict(name='predict_2048', kind='predict', members=5, samples=2048, steps=1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(['step'] * 7 + ['reload', 'forces', 'train', 'predict'])
    if kind == 'step':
        system = rng.choice(['fluid', 'fluid', 'rbc', 'channel', 'ensemble', 'poiseuille', 'random_flux'])
        if system == 'fluid':
            return dict(kind=kind, system=system, L=round(_log(rng, 6.0, 48.0), 2), rho=rng.choice([3.0, 4.0]),
                        species=rng.choice([1, 1, 2, 3, 10]), steps=rng.randint(2, 8))
        if system == 'rbc':
            L = round(_log(rng, 10.0, 28.0), 2)
            return dict(kind=kind, system=system, L=L, diameter=round(rng.uniform(4.5, min(8.0, 0.45 * L)), 2),
                        steps=rng.randint(2, 8))
        if system == 'channel':
            L = float(rng.randint(50, 64))
            return dict(kind=kind, system=system, L=L, W=float(rng.randint(25, 32)),
                        H=float(rng.randint(20, 32)), cells=rng.randint(1, 16), steps=rng.randint(1, 4))
        if system == 'ensemble':
            return dict(kind=kind, system=system, replicas=int(_log(rng, 3, 100)), steps=rng.randint(2, 8))
        if system == 'poiseuille':
            return dict(kind=kind, system=system, L=round(_log(rng, 8.0, 40.0), 2), rho=4.0, species=1,
                        steps=1)
        return dict(kind=kind, system=system, L=round(_log(rng, 8.0, 30.0), 2), rho=3.0,
                    species=rng.choice([1, 2, 10]), steps=rng.randint(1, 3))
    if kind == 'reload':
        return dict(kind=kind, system='rbc', L=round(_log(rng, 10.0, 28.0), 2), diameter=5.0, steps=1)
    if kind == 'forces':
        rho = rng.choice([3.0, 4.0])
        return dict(kind=kind, system='fluid', L=round(_log(rng, 5.5, 15.9), 2), rho=rho,
                    species=rng.randint(1, 4), steps=1)
    if kind == 'train':
        return dict(kind=kind, members=rng.randint(1, 8), samples=int(_log(rng, 300, 4500)),
                    steps=rng.randint(1, 3))
    return dict(kind=kind, members=rng.randint(2, 8), samples=int(_log(rng, 30, 20000)), steps=1)


# ---------------------------------------------------------------- inputs

def _systems(case, seed):
    """The replicas of a case (the workload generators' descriptions)."""
    system = case['system']
    if system == 'fluid':
        d = W.fluid_box(L=case['L'], rho=case['rho'], n_species=case['species'], seed=seed)
        if case['species'] > 1:
            d['kappa'][...] = np.linspace(0.5, 2.0, case['species'], dtype=np.float32)
        return [d]
    if system == 'random_flux':
        d = W.fluid_box(L=case['L'], rho=case['rho'], n_species=case['species'], seed=seed)
        d['random_flux'] = dict(m_s=0.05, rho=case['rho'])
        return [d]
    if system == 'rbc':
        return [W.single_rbc(L=case['L'], diameter=case['diameter'], seed=seed)]
    if system == 'channel':
        return [W.rbc_channel(Lx=case['L'], Ly=case['W'], H=case['H'], n_rbc=case['cells'], seed=seed)]
    if system == 'ensemble':
        # one set of boxes and cells, its particles drawn anew from the seed
        ds, rng = W.replica_ensemble(n_rep=case['replicas']), np.random.default_rng(seed)
        for d in ds:
            p, d['seed'] = d['particles'], int(rng.integers(1, 2 ** 62))
            conc = p['conc']
            d['particles'] = dict(W.fluid_particles(rng, d['L'], d['rho'], 1), conc=conc)
            for r in d['rbcs']:
                r['vel'] = rng.normal(0.0, 1.0, r['vel'].shape).astype(np.float32)
        return ds
    return [W.double_poiseuille(L=case['L'], rho=case['rho'], f=0.2, seed=seed)]


def _points(case, seed):
    """Training points of the surrogate: permeability, body force, volume
    fraction and diffusivity, with smooth positive outcomes."""
    rng = np.random.default_rng(seed)

    def x(n):
        return np.stack([10.0 ** rng.uniform(-2.0, 0.0, n), rng.uniform(0.0, 0.1, n), rng.uniform(0.0, 0.2, n),
                         10.0 ** rng.uniform(math.log10(0.3), math.log10(3.0), n)], 1).astype(np.float32)

    n = case['samples']
    X = x(n if case['kind'] == 'train' else 512)
    Y = np.stack([2.0 + X[:, 0] * (1 + 3 * X[:, 2]) + 0.1 * X[:, 3], 3.0 + np.sin(5 * X[:, 1]) + 0.3 * X[:, 3]], 1)
    return WS.init_params(seed, case['members']), X, Y.astype(np.float32), x(n)


@functools.lru_cache(maxsize=None)
def _stream():
    """One stream for all the work of the program."""
    return torch.cuda.Stream()


class _Sim:
    """A committed handle and the device arrays its state is read into."""

    def __init__(self, case, seed):
        descs = _systems(case, seed)
        self.ns = int(descs[0]['n_species'])
        if len(descs) == 1:
            self.h = bd.create_from(descs[0], stream_ptr=_stream().cuda_stream)
        else:
            parts = [bd.create_from(d) for d in descs]
            self.h = bd.tdpd_batch_create(parts)
            for p in parts:
                bd.tdpd_destroy(p)
            bd.tdpd_set_stream(self.h, _stream().cuda_stream)
        bd.tdpd_commit(self.h)
        n = [W.n_particles(d) for d in descs]
        self.pos = torch.empty(sum(n), 3, device='cuda')
        self.vel = torch.empty(sum(n), 3, device='cuda')
        self.conc = torch.empty(sum(n), self.ns, device='cuda')
        at = np.concatenate([[0], np.cumsum(n)[:-1]])
        self.ptrs = [(r, self.pos[int(a):].data_ptr(), self.vel[int(a):].data_ptr(), self.conc[int(a):].data_ptr())
                     for r, a in enumerate(at)]
        self.steps = case['steps']
        if case['kind'] == 'reload':
            s = W.flat_state(_systems(case, seed + 500)[0])[:3]
            self.host = [torch.from_numpy(a).pin_memory().numpy() for a in s]
        bd.tdpd_sync(self.h)

    def read(self):
        for r, p, v, c in self.ptrs:
            bd.tdpd_read_state_device(self.h, r, p, v, c)
        return dict(pos=self.pos, vel=self.vel, conc=self.conc)

    def __del__(self):
        if getattr(self, 'h', None):
            bd.tdpd_destroy(self.h)
            self.h = None


class _Net:
    def __init__(self, case, seed):
        params, X, Y, self.new = _points(case, seed)
        self.members, self.steps = case['members'], case['steps']
        self.h = bd.tdpd_mlp_create(self.members)
        bd.tdpd_mlp_set_params(self.h, params)
        bd.tdpd_mlp_set_data(self.h, X, Y)

    def __del__(self):
        if getattr(self, 'h', None):
            bd.tdpd_mlp_destroy(self.h)
            self.h = None


def prepare(case, seed):
    kind = case['kind']
    if kind in ('train', 'predict'):
        return kind, _Net(case, seed)
    if kind == 'forces':
        d = _systems(case, seed)[0]
        pos, vel, conc, typ, _ = W.flat_state(d)
        n = pos.shape[0]
        T, S = int(d['n_types']), int(d['n_species'])
        coef = np.stack([d['a'], d['gamma'], d['sigma']], -1).reshape(T, T, 3)
        dev = [torch.from_numpy(a).cuda() for a in (pos, vel, conc, typ)]
        out = dict(force=torch.empty(n, 3, device='cuda'), flux=torch.empty(n, S, device='cuda'))
        return kind, (bd.config_from(d), coef, d['kappa'], n, dev, out)
    return kind, _Sim(case, seed)


def run(state):
    kind, s = state
    if kind == 'step':
        bd.tdpd_step(s.h, s.steps)
        return s.read()
    if kind == 'reload':
        bd.tdpd_set_states(s.h, *s.host)
        bd.tdpd_step(s.h, s.steps)
        o = bd.tdpd_read_observables(s.h, 0)
        return dict(s.read(), kT=o['kT'], mass=[float(m) for m in o['mass']],
                    mass_membrane=[float(m) for m in o['mass_membrane']])
    if kind == 'forces':
        cfg, coef, kappa, n, dev, out = s
        bd.tdpd_pair_forces_noalloc(cfg, coef, kappa, n, *[a.data_ptr() for a in dev], 7,
                                    out['force'].data_ptr(), out['flux'].data_ptr(), _stream().cuda_stream)
        return out
    if kind == 'train':
        loss = bd.tdpd_mlp_train(s.h, s.steps, 3e-3, s.members)
        return dict(params=bd.tdpd_mlp_get_params(s.h, s.members), loss=loss.astype(np.float32))
    mean, spread, each = bd.tdpd_mlp_predict(s.h, s.new, s.members)
    return dict(mean=mean, spread=spread, each=each)


# ------------------------------------------------------------------ work

def _particles(case):
    """Expected particles and membranes of a case."""
    system = case['system']
    if system in ('fluid', 'random_flux', 'poiseuille'):
        return case['rho'] * case['L'] ** 3, 0
    if system == 'rbc':
        return 3.0 * case['L'] ** 3 + 500, 1
    if system == 'channel':
        return 3.0 * case['L'] * case['W'] * (case['H'] + 3.16) + 500 * case['cells'], case['cells']
    side3 = sum(s ** 3 for s in range(8, 17)) / 9.0
    return case['replicas'] * (3.0 * side3 + 500 * 1.8), 1.8 * case['replicas']


def work(case):
    """One pass. Bytes: each step reads and writes every particle's position,
    velocity, force, concentrations and fluxes once. Operations: each pair
    inside a cut-off once (20 + 4 (species - 1) for the flux, 110 for a
    force with its random number), 1200 per membrane bond."""
    if case['kind'] in ('train', 'predict'):
        n, m = case['samples'], case['members']
        macs = 4 * 64 + 64 * 64 + 64 * 2
        if case['kind'] == 'train':
            return dict(bytes=24.0 * n + m * 4610 * 32.0 * case['steps'], flops=6.0 * macs * n * m * (case['steps'] + 1))
        return dict(bytes=16.0 * n + m * (4610 * 4 + 8.0 * n) + 16.0 * n, flops=2.0 * macs * n * m)
    n, cells = _particles(case)
    ns = 2 if case['system'] == 'channel' else case.get('species', 1)
    rho = case.get('rho', 3.0)
    rc = 1.58 if case['system'] == 'poiseuille' else 1.0
    sphere = 4.0 / 3.0 * math.pi * rho
    flux = 0.5 * sphere * 1.58 ** 3 * (20 + 4 * (ns - 1))
    if case['system'] == 'random_flux':
        flux += 0.5 * sphere * 1.58 ** 3 * (110 * ((ns + 1) // 2) + 8 * ns)
    ops = n * (flux + 0.5 * sphere * rc ** 3 * 110) + cells * 1494 * 1200.0
    evals = case['steps'] + (1 if case['kind'] == 'reload' else 0)
    state = n * (36 + 8 * ns)
    if case['kind'] == 'forces':
        return dict(bytes=n * (12.0 + 12 + 4 * ns + 4 + 12 + 4 * ns), flops=ops)
    return dict(bytes=2.0 * state * evals, flops=ops * evals)


# ----------------------------------------------------------------- exact

F64 = dict(dtype=torch.float64, device='cuda')
M32 = 0xFFFFFFFF


def _t(a):
    return torch.as_tensor(np.asarray(a, np.float64), **F64)


def _normals(i, j, seed, step, stream):
    """Box-Muller normals (cosine, sine branch) of eight TEA rounds on the
    block (min id, max id) under the key (seed, step, stream)."""
    y, z = torch.minimum(i, j), torch.maximum(i, j)
    k0, k1 = seed & M32, (seed >> 32) & M32
    k2, k3 = step & M32, stream & M32
    s = 0
    for _ in range(8):
        s = (s + 0x9E3779B9) & M32
        y = (y + (((z << 4) + k0) ^ (z + s) ^ ((z >> 5) + k1))) & M32
        z = (z + (((y << 4) + k2) ^ (y + s) ^ ((y >> 5) + k3))) & M32
    u1 = (y >> 9).double() * 2.0 ** -23 + 2.0 ** -24
    u2 = (z >> 9).double() * 2.0 ** -23 + 2.0 ** -24
    r = torch.sqrt(-2.0 * torch.log(u1))
    return r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)


def _pairs(x, L, periodic, rcut):
    """Every unordered pair closer than rcut: i, j, x_i - x_j, |x_i - x_j|."""
    n = x.shape[0]
    nc = [int(math.floor(l / rcut)) for l in L]
    size = torch.as_tensor([l / c for l, c in zip(L, nc)], **F64)
    c = torch.minimum((x / size).long(), torch.as_tensor([k - 1 for k in nc], device='cuda')).clamp_(min=0)
    cell = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
    ncell = nc[0] * nc[1] * nc[2]
    order = torch.argsort(cell)
    count = torch.bincount(cell, minlength=ncell)
    cap = int(count.max())
    start = torch.cumsum(count, 0) - count
    rank = torch.arange(n, device='cuda') - start[cell[order]]
    table = torch.full((ncell + 1, cap), -1, dtype=torch.long, device='cuda')
    table[cell[order], rank] = order
    cells = torch.arange(ncell, device='cuda')
    cx, cy, cz = cells % nc[0], (cells // nc[0]) % nc[1], cells // (nc[0] * nc[1])
    Lt = torch.as_tensor(L, **F64)
    half = [(0, 0, 0)] + [(a, b, e) for e in (-1, 0, 1) for b in (-1, 0, 1) for a in (-1, 0, 1) if (e, b, a) > (0, 0, 0)]
    dx, dy, dz = (torch.as_tensor([o[q] for o in half], device='cuda')[:, None] for q in range(3))
    z = cz + dz
    nb = ((z % nc[2]) * nc[1] + (cy + dy) % nc[1]) * nc[0] + (cx + dx) % nc[0]
    if not periodic[2]:
        nb = torch.where((z >= 0) & (z < nc[2]), nb, torch.full_like(nb, ncell))
    nb = nb.reshape(-1)
    here = cells.repeat(len(half))
    upper = torch.ones(cap, cap, dtype=torch.bool, device='cuda').triu(1)
    found = []
    chunk = max(1, (1 << 25) // (cap * cap))
    for k in range(0, nb.shape[0], chunk):
        a, b = table[here[k:k + chunk]], table[nb[k:k + chunk]]
        ok = (a[:, :, None] >= 0) & (b[:, None, :] >= 0)
        own = max(0, min(ncell - k, chunk))         # rows that pair a cell with itself
        ok[:own] &= upper
        r2 = torch.zeros(ok.shape, **F64)
        for q in range(3):
            d = x[a.clamp(min=0), q][:, :, None] - x[b.clamp(min=0), q][:, None, :]
            if periodic[q]:
                d = d - L[q] * torch.round(d / L[q])
            r2 += d * d
        m, p, q = torch.nonzero(ok & (r2 < rcut * rcut), as_tuple=True)
        found.append(torch.stack([a[m, p], b[m, q]]))
    i, j = torch.cat(found, 1)
    d = x[i] - x[j]
    per = torch.as_tensor([float(p) for p in periodic], **F64)
    d = d - per * Lt * torch.round(d / Lt)
    return i, j, d, d.norm(dim=1)


class _Exact:
    """One replica in binary64: forces, fluxes and the velocity-Verlet step."""

    def __init__(self, d):
        self.d = d
        self.L = [float(v) for v in d['L']]
        self.periodic = [int(v) for v in d['periodic']]
        pos, vel, conc, typ, body = W.flat_state(d)
        self.x, self.v, self.c = _t(pos), _t(vel), _t(conc)
        self.type = torch.as_tensor(typ, device='cuda').long()
        self.body = torch.as_tensor(body, device='cuda').long()
        self.frozen = ((int(d['frozen_types']) >> self.type) & 1).bool()
        self.tab = {k: _t(d[k]) for k in ('a', 'gamma', 'sigma', 'kappa')}
        self.num = {k: float(d[k]) for k in ('dt', 'lam', 'rc', 'rcc', 's_f', 's_c', 'wall_lo', 'wall_hi')}
        self.mem = [self._membrane(b) for b in range(len(d['rbcs']))]
        self.step = 0

    def _membrane(self, b):
        d, m = self.d, self.d['membrane']
        r = d['rbcs'][b]
        tri = torch.as_tensor(r['tri'], device='cuda').long()
        e = torch.cat([tri[:, [0, 1]], tri[:, [1, 2]], tri[:, [2, 0]]])
        apex = torch.cat([tri[:, 2], tri[:, 0], tri[:, 1]])
        nv = r['pos'].shape[0]
        key, rev = e[:, 0] * nv + e[:, 1], e[:, 1] * nv + e[:, 0]
        order = torch.argsort(key)
        other = apex[order[torch.searchsorted(key[order], rev)]]
        fwd = e[:, 0] < e[:, 1]
        q = torch.stack([e[fwd, 0], e[fwd, 1], apex[fwd], other[fwd]])       # a, b, c (left), d (right)
        rest = self._unwrap(_t(r['pos'] if r['rest'] is None else r['rest']))
        l0 = (rest[q[0]] - rest[q[1]]).norm(dim=1)
        A, V = self._areas(rest, tri)
        x0, mm = float(np.float32(m['x0'])), float(np.float32(m['m']))
        kT, p = float(np.float32(m['kT'])), float(np.float32(m['p']))
        kp = kT / p * (0.25 / (1 - x0) ** 2 - 0.25 + x0) * l0 ** mm
        A0 = A.sum()
        v_ratio = float(np.float32(m['v_ratio']))
        return dict(tri=tri, q=q, lm=l0 / x0, kp=kp, a0=A, A0=A0, V0=v_ratio * A0 ** 1.5 if v_ratio > 0 else V)

    def _unwrap(self, x):
        L = torch.as_tensor(self.L, **F64)
        t = x * (2 * math.pi / L)
        ref = torch.atan2(torch.sin(t).mean(0), torch.cos(t).mean(0)) * L / (2 * math.pi)
        per = torch.as_tensor([float(p) for p in self.periodic], **F64)
        ref = torch.where(per > 0, ref, x.mean(0))
        return x - per * L * torch.round((x - ref) / L)

    @staticmethod
    def _areas(x, tri):
        p0, p1, p2 = x[tri[:, 0]], x[tri[:, 1]], x[tri[:, 2]]
        A = 0.5 * torch.linalg.cross(p1 - p0, p2 - p0).norm(dim=1)
        o = x.detach().mean(0)
        return A, ((p0 - o) * torch.linalg.cross(p1 - o, p2 - o)).sum() / 6.0

    def _membrane_force(self, M, x, v, ids, step):
        m = {k: float(np.float32(w)) for k, w in self.d['membrane'].items()}
        x = self._unwrap(x).requires_grad_(True)
        A, V = self._areas(x, M['tri'])
        a, b, c, d = (x[k] for k in M['q'])
        n1, n2 = torch.linalg.cross(b - a, c - a), torch.linalg.cross(a - b, d - b)
        e = (b - a) / (b - a).norm(dim=1, keepdim=True)
        inv = 1.0 / (n1.norm(dim=1) * n2.norm(dim=1))
        cos, sin = (n1 * n2).sum(1) * inv, (torch.linalg.cross(n1, n2) * e).sum(1) * inv
        U = (m['kg'] * (A.sum() - M['A0']) ** 2 / (2 * M['A0']) + m['kv'] * (V - M['V0']) ** 2 / (2 * M['V0'])
             + (m['kl'] * (A - M['a0']) ** 2 / (2 * M['a0'])).sum()
             - m['kb'] * (cos * math.cos(m['theta0']) + sin * math.sin(m['theta0'])).sum())
        f = -torch.autograd.grad(U, x)[0]
        x = x.detach()
        i, j = M['q'][0], M['q'][1]
        r = x[i] - x[j]
        l = r.norm(dim=1, keepdim=True)
        e = r / l
        y = l / M['lm'][:, None]
        fb = -(m['kT'] / m['p'] * (0.25 / (1 - y) ** 2 - 0.25 + y) - M['kp'][:, None] / l ** m['m']) * e
        vij = v[i] - v[j]
        fb = fb - m['gammaT'] * vij - m['gammaC'] * (vij * e).sum(1, keepdim=True) * e
        z = []
        for s in range(5):
            z += _normals(ids[i], ids[j], int(self.d['seed']), step, 1 + s)
        Z = torch.stack(z[:9], 1).reshape(-1, 3, 3)
        tr = Z.diagonal(dim1=1, dim2=2).sum(1)[:, None]
        we = torch.einsum('nij,nj->ni', 0.5 * (Z + Z.transpose(1, 2)), e) - tr / 3 * e
        s0 = math.sqrt(2 * m['kT'] / self.num['dt'])
        fb = fb + s0 * (math.sqrt(2 * m['gammaT']) * we + math.sqrt(3 * m['gammaC'] - m['gammaT']) / 3 * tr * e)
        return f.index_add(0, i, fb).index_add(0, j, -fb)

    def forces(self, x, v, c, step, membranes=True):
        d, num = self.d, self.num
        F, Q = torch.zeros_like(x), torch.zeros_like(c)
        i, j, dr, r = _pairs(x, self.L, self.periodic, max(num['rc'], num['rcc']))
        ti, tj = self.type[i], self.type[j]
        k = torch.nonzero(r < num['rcc'])[:, 0]
        wdc = (1 - r[k] / num['rcc']) ** num['s_c']
        kap = self.tab['kappa'][ti[k], tj[k]]
        q = -kap * wdc[:, None] * (c[i[k]] - c[j[k]])
        flux = d.get('random_flux')
        if flux:
            m_s, rho = float(np.float32(flux['m_s'])), float(np.float32(flux['rho']))
            amp = m_s * math.sqrt(rho) * torch.sqrt(wdc / num['dt']) * torch.where(i[k] < j[k], 1.0, -1.0).double()
            for s in range(c.shape[1]):
                z = _normals(i[k], j[k], int(d['seed']), step, 6 + s // 2)[s % 2]
                q[:, s] += amp * torch.sqrt((kap[:, s] * (c[i[k], s] + c[j[k], s])).clamp(min=0)) * z
        Q.index_add_(0, i[k], q)
        Q.index_add_(0, j[k], -q)
        near = r < num['rc']
        if d['exclude_same_body']:
            near &= ~((self.body[i] >= 0) & (self.body[i] == self.body[j]))
        k = torch.nonzero(near)[:, 0]
        i, j, ti, tj, dr, r = i[k], j[k], ti[k], tj[k], dr[k], r[k]
        e = dr / r[:, None]
        w = 1 - r / num['rc']
        wr = w ** (0.5 * num['s_f'])
        xi = _normals(i, j, int(d['seed']), step, 0)[0]
        f = (self.tab['a'][ti, tj] * w - self.tab['gamma'][ti, tj] * wr * wr * (e * (v[i] - v[j])).sum(1)
             + self.tab['sigma'][ti, tj] * wr * xi / math.sqrt(num['dt']))[:, None] * e
        F.index_add_(0, i, f)
        F.index_add_(0, j, -f)
        if membranes:
            for b, M in enumerate(self.mem):
                ids = torch.nonzero(self.body == b)[:, 0]
                F[ids] += self._membrane_force(M, x[ids], v[ids], ids, step)
        body = _t(d['body_force']).expand_as(F).clone()
        if d.get('body_force_flip'):
            body[x[:, 2] >= 0.5 * self.L[2]] *= -1
        body[self.frozen] = 0
        F += body
        re = d.get('reaction')
        if re:
            rate = float(np.float32(re['k'])) * c[:, re['src']] * ((int(re['types']) >> self.type) & 1)
            Q[:, re['src']] -= rate
            Q[:, re['dst']] += rate
        return F, Q

    def start(self):
        self.F, self.Q = self.forces(self.x, self.v, self.c, self.step)
        return self

    def advance(self, steps):
        num = self.num
        dt, lam, move = num['dt'], num['lam'], (~self.frozen)[:, None]
        Lt = torch.as_tensor(self.L, **F64)
        for _ in range(steps):
            self.step += 1
            x = self.x + dt * self.v + 0.5 * dt * dt * self.F
            v = self.v
            for q in range(3):
                if self.periodic[q]:
                    continue
                low, high = x[:, q] < num['wall_lo'], x[:, q] > num['wall_hi']
                x[:, q] = torch.where(low, 2 * num['wall_lo'] - x[:, q], torch.where(high, 2 * num['wall_hi'] - x[:, q], x[:, q]))
                v = torch.where((low | high)[:, None], -v, v)
            per = torch.as_tensor([float(p) for p in self.periodic], **F64)
            x = x - per * Lt * torch.floor(x / Lt)
            x = torch.where(move, x, self.x)
            v = torch.where(move, v, self.v)
            vt = torch.where(move, v + lam * dt * self.F, v)
            ct = torch.where(move, self.c + lam * dt * self.Q, self.c)
            F, Q = self.forces(x, vt, ct, self.step)
            self.v = torch.where(move, v + 0.5 * dt * (self.F + F), v)
            self.c = torch.where(move, self.c + 0.5 * dt * (self.Q + Q), self.c)
            self.x, self.F, self.Q = x, F, Q
        return self


def _exact_net(case, seed):
    params, X, Y, new = _points(case, seed)
    st = [(a.astype(np.float64).mean(0), a.astype(np.float64).std(0) + 1e-12) for a in (X, Y)]

    def scaled(a, k):
        return _t(((a - st[k][0]) / st[k][1]).astype(np.float32))

    def net(p, x):
        w = p.to(torch.bfloat16).double()
        w = w.detach().requires_grad_(True)
        at, parts = 0, []
        for sh in WS.SHAPES:
            n = int(np.prod(sh))
            parts.append(w[:, at:at + n].reshape((-1,) + tuple(sh)))
            at += n
        W1, b1, W2, b2, W3, b3 = parts
        h = torch.nn.functional.gelu(torch.einsum('moi,ni->mno', W1, x) + b1[:, None])
        h = torch.nn.functional.gelu(torch.einsum('moi,mni->mno', W2, h) + b2[:, None])
        return w, torch.einsum('moi,mni->mno', W3, h) + b3[:, None]

    p = _t(params)
    if case['kind'] == 'predict':
        with torch.no_grad():
            y = net(p, scaled(new, 0))[1] * _t(st[1][1]) + _t(st[1][0])
        mean = y.mean(0)
        return dict(mean=mean, spread=y.std(0) / mean.abs(), each=y)
    x, t = scaled(X, 0), scaled(Y, 1)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    lr, b1, b2 = float(np.float32(3e-3)), 0.9, 0.999
    for k in range(1, case['steps'] + 2):
        w, y = net(p, x)
        loss = ((y - t) ** 2).mean((1, 2))
        if k > case['steps']:
            # the loss jumps where a bfloat16 rounding of an updated weight
            # flips with its last bits: it has no value to be held to
            return dict(params=p.detach(), loss=None)
        g = torch.autograd.grad(loss.sum(), w)[0]
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        p = p - lr * (m / (1 - b1 ** k)) / (torch.sqrt(v / (1 - b2 ** k)) + 1e-8)


def exact(case, seed):
    kind = case['kind']
    if kind in ('train', 'predict'):
        return _exact_net(case, seed)
    if kind == 'forces':
        e = _Exact(_systems(case, seed)[0])
        F, Q = e.forces(e.x, e.v, e.c, 7)
        return dict(force=F, flux=Q)
    if kind == 'reload':
        e = _Exact(_systems(case, seed)[0])
        e.x, e.v, e.c = (_t(a) for a in W.flat_state(_systems(case, seed + 500)[0])[:3])
        e.start().advance(case['steps'])
        vm = e.v - e.v.mean(0)
        mem = e.body >= 0
        return dict(pos=e.x, vel=e.v, conc=e.c, kT=float((vm * vm).sum() / (3 * (e.x.shape[0] - 1))),
                    mass=[float(s) for s in e.c.sum(0)], mass_membrane=[float(s) for s in e.c[mem].sum(0)])
    es = [_Exact(d).start().advance(case['steps']) for d in _systems(case, seed)]
    return dict(pos=torch.cat([e.x for e in es]), vel=torch.cat([e.v for e in es]), conc=torch.cat([e.c for e in es]))
