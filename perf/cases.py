"""What a user of this library has it do, as cases whose time and outputs can be measured.

A case is a dict of plain values with a ``kind``:

* ``suspension`` -- a dense suspension settling in a periodic box, equal or
  unequal spheres, optionally with no-slip walls at the z faces; a pass is a
  number of time steps and the read-out of the particle state (the fluid and
  its flags too in small boxes; the fields of a large box are a gigabyte on
  the host and are written out once in thousands of steps).
* ``wall`` -- one sphere falling towards a no-slip wall in a small box
  (the sphere-wall workload and the boxes of the batched one), with fields.
* ``stokes`` -- a fixed sphere in a periodic box driven by a body force (the
  Stokes array of the validation), with fields.
* ``shear`` -- a fixed sphere near the resting wall of a shear flow (the drag
  and lift validation); the forces are read.
* ``probe`` -- a sphere whose velocity the caller sets before every step and a
  density probe moving with it (the settling validation): one host round trip
  per step.
* ``batch`` -- several sphere-wall boxes advanced together in batches on their
  own streams.
* ``map`` -- the sphere-to-cell mapping into buffers of the caller.

The state getters return float64 arrays whatever the PDF storage; a pass hands
them on in the precision that the run computes in (float64 for float64
storage, float32, float16 or bfloat16 for those storages), except positions,
which every storage keeps in float64 and a pass hands on in float32 below it.
:func:`exact` restates one pass in plain float64 torch.
"""
import math

import numpy as np
import torch

from paper_2003_01490_gb300 import lbmdem as L
from paper_2003_01490_gb300 import tune

# the largest box whose fields a pass reads (cells)
FIELDS_MAX = 600_000


def _suspension(name, nx, ny, nz, n, d, storage, steps, spread=0.0, walls=False):
    return dict(name=name, kind='suspension', nx=nx, ny=ny, nz=nz, n=n, d=d, spread=spread, storage=storage,
                steps=steps, walls=walls)


def listed():
    return [
        # the sphere-wall workload: the smallest box, float64, latency of a step
        dict(name='wall_f64_32x32x64', kind='wall', nx=32, ny=32, nz=64, d=8.0, storage='f64', tau=0.6,
             ratio=8.0, steps=100),
        # one box of the batched workload run alone in float32
        dict(name='wall_f32_40x40x80', kind='wall', nx=40, ny=40, nz=80, d=10.0, storage='f32', tau=0.57,
             ratio=3.0, steps=100),
        # the Stokes array of the validation
        dict(name='stokes_f64_40', kind='stokes', nx=40, ny=40, nz=40, d=20.0, storage='f64', tau=0.7, steps=100),
        # prescribed motion with a density probe: a host round trip per step
        dict(name='probe_f32_80x80x160', kind='probe', nx=80, ny=80, nz=160, d=20.0, storage='f32', steps=20,
             probes=1),
        # drag and lift near a wall at half resolution: fluid only but for one sphere
        dict(name='shear_f32_480x160x80', kind='shear', nx=480, ny=160, nz=80, d=10.0, storage='f32', steps=50),
        # the reduced suspension of the parity runs
        _suspension('suspension_f32_64x64x128', 64, 64, 128, 150, 12.0, 'f32', 50),
        # a suspension job of the served stream in its default storage
        _suspension('suspension_f16_192', 192, 192, 192, 2000, 12.0, 'f16', 20),
        # odd sides, unequal spheres, walls, bfloat16
        _suspension('channel_bf16_131x97x203', 131, 97, 203, 500, 12.0, 'bf16', 20, spread=0.3, walls=True),
        # the profiled suspension
        _suspension('suspension_f32_128x128x256', 128, 128, 256, 1250, 12.0, 'f32', 20),
        # the headline suspension: the largest
        _suspension('suspension_f32_256x256x512', 256, 256, 512, 10000, 12.0, 'f32', 10),
        # many small boxes at once
        dict(name='batch_f32_16', kind='batch', boxes=16, smin=32, smax=96, groups=4, storage='f32', steps=20),
        # mapping 10,000 spheres without a device allocation
        dict(name='map_256x256x512', kind='map', nx=256, ny=256, nz=512, n=10000, d=12.0, spread=0.0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(['suspension', 'suspension', 'suspension', 'wall', 'stokes', 'probe', 'shear', 'batch', 'map'])
    if kind in ('suspension', 'map'):
        nx, ny, nz = log_int(48, 256), log_int(48, 256), log_int(48, 384)
        d = round(rng.uniform(8.0, 16.0), 2)
        spread = rng.choice([0.0, 0.0, 0.3])
        phi = rng.uniform(0.02, 0.27)
        n = max(1, min(10000, int(phi * nx * ny * nz / (math.pi / 6.0 * (d * (1.0 + 0.5 * spread)) ** 3))))
        if kind == 'map':
            return dict(kind='map', nx=nx, ny=ny, nz=nz, n=n, d=d, spread=spread)
        return dict(kind='suspension', nx=nx, ny=ny, nz=nz, n=n, d=d, spread=spread,
                    storage=rng.choice(['f32', 'f32', 'f16', 'bf16']), steps=20, walls=rng.random() < 0.3)
    if kind == 'wall':
        s = rng.randrange(32, 97)
        return dict(kind='wall', nx=s, ny=rng.randrange(32, 97), nz=2 * s, d=round(min(24.0, max(8.0, s / 4.0)), 2),
                    storage=rng.choice(['f64', 'f32', 'f16']), tau=round(rng.uniform(0.52, 0.8), 3),
                    ratio=round(rng.uniform(1.5, 10.0), 2), steps=50)
    if kind == 'stokes':
        n = rng.randrange(24, 65)
        return dict(kind='stokes', nx=n, ny=n, nz=n, d=round(0.5 * n, 2), storage=rng.choice(['f64', 'f64', 'f32']),
                    tau=round(rng.uniform(0.55, 1.5), 3), steps=50)
    if kind == 'probe':
        d = rng.randrange(8, 25)
        return dict(kind='probe', nx=4 * d, ny=4 * d + rng.randrange(3), nz=8 * d, d=float(d),
                    storage=rng.choice(['f64', 'f32']), steps=20, probes=rng.choice([1, 1, 16]))
    if kind == 'shear':
        d = rng.randrange(6, 13)
        return dict(kind='shear', nx=48 * d + rng.randrange(32), ny=16 * d, nz=8 * d, d=float(d),
                    storage=rng.choice(['f32', 'f16']), steps=20)
    return dict(kind='batch', boxes=rng.randrange(2, 25), smin=32, smax=rng.choice([48, 64, 96]),
                groups=rng.choice([1, 2, 4]), storage=rng.choice(['f32', 'f16']), steps=20)


# ---------------------------------------------------------------- inputs

def _radii(case, rng):
    return 0.5 * case['d'] * (1.0 + case['spread'] * (rng.random(case['n']) - 0.5))


def _place(case, radius, rng, walls):
    """Centres of non-overlapping spheres by random sequential addition, tried
    a block at a time: a try stands if it overlaps no sphere placed before and
    no earlier try of its block. Radii are put in the order of placement."""
    n, dev = len(radius), 'cuda' if torch.cuda.is_available() else 'cpu'
    shape = torch.tensor([case['nx'], case['ny'], case['nz']], dtype=torch.float64, device=dev)
    nb = (shape / (2.0 * radius.max())).floor().long().clamp(min=1)
    cap = 16
    table = torch.full((int(nb.prod()), cap), -1, device=dev)
    count = torch.zeros(int(nb.prod()), dtype=torch.int64, device=dev)
    pos = torch.zeros((n, 3), dtype=torch.float64, device=dev)
    rad = torch.as_tensor(radius, device=dev).clone()
    near = torch.tensor([[a, b, c] for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)], device=dev)
    wraps = torch.tensor([1.0, 1.0, 0.0 if walls else 1.0], dtype=torch.float64, device=dev)

    def apart(x, y, reach):
        e = x - y
        e = e - wraps * shape * (e / shape).round()
        return (e * e).sum(-1) >= reach * reach

    def bin_of(b):
        return (b[..., 2] * nb[1] + b[..., 1]) * nb[0] + b[..., 0]

    done = 0
    for _ in range(4000):
        if done == n:
            break
        m = min(1024, max(64, 4 * (n - done)))
        # the next spheres, each tried several times when few are left
        want = done + torch.arange(m, device=dev) % (n - done)
        x = torch.as_tensor(rng.random((m, 3)), device=dev)
        r = rad[want]
        low = r[:, None] * (1.0 - wraps) + 1e-6
        x = low + x * (shape - 2.0 * low)
        b = torch.minimum((x / (shape / nb)).long(), nb - 1)
        other = table[bin_of((b[:, None, :] + near) % nb)].reshape(m, -1)
        ok = (apart(x[:, None, :], pos[other], r[:, None] + rad[other]) | (other < 0)).all(1)
        x, want, b, r = x[ok], want[ok], b[ok], r[ok]
        if not len(x):
            continue
        clash = ~apart(x[:, None, :], x[None], r[:, None] + r[None]) | (want[:, None] == want[None])
        ok = ~torch.tril(clash, -1).any(1)
        x, want, b = x[ok], want[ok], bin_of(b[ok])
        k = len(x)
        left = torch.ones(n, dtype=torch.bool, device=dev)
        left[:done] = False
        left[want] = False
        rad[done:] = torch.cat([rad[want], rad[left]])
        slot = count[b] + torch.tril(b[:, None] == b[None], -1).sum(1)
        if int(slot.max()) >= cap:
            raise RuntimeError('placement table is full')
        table[b, slot] = done + torch.arange(k, device=dev)
        count.index_add_(0, b, torch.ones_like(b))
        pos[done:done + k] = x
        done += k
    if done < n:
        raise RuntimeError('no room for %d spheres' % n)
    radius[:] = rad.cpu().numpy()
    return pos.cpu().numpy()


def _settling_gravity(nu, u, ratio, d):
    """g of a sphere of density ratio that settles at u (Schiller-Naumann balance)."""
    return 18.0 * nu * u * (1.0 + 0.15 * (u * d / nu) ** 0.687) / ((ratio - 1.0) * d * d)


def _setup(case, seed):
    """Box, parameters and spheres of one simulation (not of a batch or map)."""
    rng = np.random.default_rng(seed)
    shape = (case['nx'], case['ny'], case['nz'])
    d = case['d']
    s = dict(shape=shape, periodic=(1, 1, 1), body=(0.0, 0.0, 0.0), gravity=0.0, counter=False, motion=L.MOTION_DEM,
             top=0.0, storage=case['storage'], flow=0.0)
    if case['kind'] == 'suspension':
        radius = _radii(case, rng)
        n = len(radius)
        pos = _place(case, radius, rng, case['walls'])
        nu = (0.55 - 0.5) / 3.0
        s.update(tau=0.55, gravity=0.005 * 18.0 * nu / (1.5 * d * d), counter=not case['walls'], pos=pos,
                 vel=rng.normal(0.0, 1e-3, (n, 3)), omega=rng.normal(0.0, 1e-4, (n, 3)), radius=radius,
                 density=np.full(n, 2.5))
        if case['walls']:
            s['periodic'] = (1, 1, 0)
        return s
    # one sphere, off the middle so that no force or torque vanishes by symmetry
    at = 0.5 * np.array(shape) + rng.uniform(-1.0, 1.0, 3)
    vel, omega, ratio = np.zeros(3), np.zeros(3), 1.0
    if case['kind'] == 'wall':
        nu = (case['tau'] - 0.5) / 3.0
        ratio = case['ratio']
        at[2] = 0.25 * shape[2] + 0.5 * d + rng.uniform(0.0, 1.0)
        vel = np.array([0.004, -0.003, -0.02]) * rng.uniform(0.8, 1.2, 3)
        omega = np.array([5e-3, -4e-3, 3e-3]) * rng.uniform(0.8, 1.2, 3)
        s.update(tau=case['tau'], periodic=(1, 1, 0), gravity=_settling_gravity(nu, 0.02, ratio, d))
    elif case['kind'] == 'stokes':
        s.update(tau=case['tau'], body=(1e-5 * rng.uniform(0.8, 1.2), 3e-6, 0.0), motion=L.MOTION_FIXED)
    elif case['kind'] == 'shear':
        gap = rng.uniform(0.505, 1.0)
        at[2] = gap * d
        rate = 0.1 / shape[2]
        s.update(tau=3.0 * rate * gap * d * d / 5.0 + 0.5, periodic=(1, 1, 0), motion=L.MOTION_FIXED, top=0.1, flow=0.1)
        omega = np.array([0.0, 1e-4, 0.0])
    else:
        ratio = 8.34
        nu = 0.02 * d / 164.0
        omega = np.array([2e-4, -1e-4, 1e-4]) * rng.uniform(0.8, 1.2, 3)
        s.update(tau=3.0 * nu + 0.5, periodic=(0, 0, 1), motion=L.MOTION_PRESCRIBED,
                 fall=18.0 * nu / (ratio * d * d), jitter=rng.uniform(-0.3, 0.3, (case['probes'], 3)))
    s.update(pos=at[None, :], vel=vel[None, :], omega=omega[None, :], radius=np.array([0.5 * d]),
             density=np.array([ratio]))
    return s


def _boxes(case, seed):
    """The boxes of a batch: sides in steps of 8 cells, spheres of a quarter of the side."""
    rng = np.random.default_rng(seed)
    sides = np.random.default_rng(case['boxes']).integers(case['smin'] // 8, case['smax'] // 8 + 1, case['boxes']) * 8
    out = []
    for s in sides:
        one = dict(kind='wall', nx=int(s), ny=int(s), nz=2 * int(s), d=float(min(24, max(8, round(s / 4)))),
                   storage=case['storage'], tau=float(rng.uniform(0.52, 0.8)), ratio=float(rng.uniform(1.5, 10.0)))
        out.append(_setup(one, int(rng.integers(1 << 31))))
    return out


def _context(s):
    r, d = L.lbm_default_params()
    r.tau = s['tau']
    d.gravity[2] = -s['gravity']
    d.fluid_counterforce = int(s['counter'])
    d.fixed_particles = s['motion']
    hi = [[0.0] * 3, [0.0] * 3, [s['top'], 0.0, 0.0]]
    ctx = L.lbm_create(L.make_grid(s['shape'], s['periodic'], wall_vel_hi=hi), r, s['body'], d, s['storage'],
                       max_particles=len(s['radius']))
    if s['flow']:
        nx, ny, nz = s['shape']
        feq = _equilibrium(torch.as_tensor(s['flow'] * (np.arange(nz) + 0.5) / nz)).numpy()
        L.lbm_set_pdfs(ctx, np.ascontiguousarray(np.broadcast_to(feq[:, :, None, None], (19, nz, ny, nx))))
    L.lbm_add_spheres(ctx, s['pos'], s['vel'], s['omega'], s['radius'], s['density'])
    return ctx


def prepare(case, seed):
    if case['kind'] == 'map':
        rng = np.random.default_rng(seed)
        radius = _radii(case, rng)
        pos = _place(case, radius, rng, False)
        shape = (case['nx'], case['ny'], case['nz'])
        cells = shape[0] * shape[1] * shape[2]
        return dict(case=case, grid=L.make_grid(shape), pos=torch.tensor(pos, device='cuda').reshape(-1),
                    radius=torch.tensor(radius, device='cuda'),
                    flags=torch.empty(cells, dtype=torch.uint8, device='cuda'),
                    owner=torch.empty(cells, dtype=torch.int32, device='cuda'))
    if case['kind'] == 'batch':
        ctxs = [_context(s) for s in _boxes(case, seed)]
        for c in ctxs:      # a batch takes instances that have stepped once
            L.lbm_step(c, 1)
        return dict(case=case, ctxs=ctxs, groups=tune.make_groups(ctxs, case['groups']))
    s = _setup(case, seed)
    state = dict(case=case, ctx=_context(s))
    if case['kind'] == 'probe':
        state.update(setup=s, t=0, x=s['pos'][0].copy())
    return state


# ---------------------------------------------------------------- one pass

TYPES = {'f64': torch.float64, 'f32': torch.float32, 'f16': torch.float16, 'bf16': torch.bfloat16}


def _out(storage, **arrays):
    """Float arrays in the precision of the run (positions at least float32)."""
    kind = TYPES[storage]
    wide = kind if kind == torch.float64 else torch.float32
    return {k: torch.from_numpy(v).to(wide if k == 'pos' else kind) for k, v in arrays.items()}


def _fall(s, t):
    """Velocity and spin set for step t of the prescribed settling, from 0.4 of its end velocity on."""
    u = -0.02 * (1.0 - math.exp(-10.0 * s['fall'] * t - 0.5))
    return np.array([[0.0, 0.0, u]]), s['omega']


def _probe_points(case, s, x):
    return x + np.array([case['d'], 0.0, 0.0]) + s['jitter']


def run(state):
    case = state['case']
    if case['kind'] == 'map':
        L.lbm_map_spheres_noalloc(state['grid'], 2.0, state['pos'], state['radius'], state['flags'], state['owner'])
        return state['flags'], state['owner']
    if case['kind'] == 'batch':
        for b, _ in state['groups']:
            L.lbm_batch_step(b, case['steps'])
        for b, _ in state['groups']:
            L.lbm_batch_sync(b)
        got = [L.lbm_get_particle_state(c) for c in state['ctxs']]
        return _out(case['storage'], **{k: np.concatenate([g[k] for g in got]) for k in got[0]})
    ctx = state['ctx']
    if case['kind'] == 'probe':
        s, rho = state['setup'], np.empty((case['steps'], case['probes']))
        for k in range(case['steps']):
            state['t'] += 1
            vel, omega = _fall(s, state['t'])
            L.lbm_set_particle_velocity(ctx, vel, omega)
            L.lbm_step(ctx, 1)
            state['x'] = (state['x'] + vel[0]) % s['shape'][2]
            rho[k] = L.lbm_sample_density(ctx, _probe_points(case, s, state['x']))
        return _out(case['storage'], rho=rho, **L.lbm_get_particle_state(ctx))
    L.lbm_step(ctx, case['steps'])
    out = _out(case['storage'], **L.lbm_get_particle_state(ctx))
    if ctx.ncells <= FIELDS_MAX and case['kind'] != 'shear':
        rho, u, flags = L.lbm_get_fields(ctx)
        out.update(_out(case['storage'], rho=rho, u=u), flags=flags)
    return out


def work(case):
    """Bytes and operations of one pass: per step every fluid cell's 19 PDFs
    read and written and a flag byte per cell; 230 operations per fluid cell
    (collision with forcing) and 75 per particle link (5.7 links per unit of
    sphere surface); the read-out once."""
    if case['kind'] == 'map':
        cells = case['nx'] * case['ny'] * case['nz']
        return {'bytes': 5 * cells + 32 * case['n'], 'flops': 9 * 729 * case['n']}
    if case['kind'] == 'batch':
        boxes = [(int(np.prod(s['shape'])), s['radius']) for s in _boxes(case, 0)]
    else:
        radius = np.full(case.get('n', 1), 0.5 * case['d'])
        boxes = [(case['nx'] * case['ny'] * case['nz'], radius)]
    es = {'f64': 8, 'f32': 4}.get(case['storage'], 2)
    total = {'bytes': 0, 'flops': 0}
    for cells, r in boxes:
        fluid = cells - float((4.0 / 3.0 * math.pi * r ** 3).sum())
        links = 5.7 * float((4.0 * math.pi * r ** 2).sum())
        total['bytes'] += case['steps'] * (fluid * 38 * es + cells) + 120 * len(r)
        total['flops'] += case['steps'] * (230 * fluid + 75 * links)
        if cells <= FIELDS_MAX and case['kind'] in ('wall', 'stokes', 'suspension'):
            total['bytes'] += fluid * 19 * es + 33 * cells
    return total


# ------------------------------------------- the same pass in plain float64

# lattice velocities and weights in the order of the paper's App. A
_C = [(0, 0, 0), (0, 1, 0), (0, -1, 0), (-1, 0, 0), (1, 0, 0), (0, 0, 1), (0, 0, -1), (-1, 1, 0), (1, 1, 0),
      (-1, -1, 0), (1, -1, 0), (0, 1, 1), (0, -1, 1), (-1, 0, 1), (1, 0, 1), (0, 1, -1), (0, -1, -1), (-1, 0, -1),
      (1, 0, -1)]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_OPP = [_C.index(tuple(-v for v in c)) for c in _C]


def _equilibrium(ux):
    """Equilibrium PDFs (density 1) of the velocities (ux, 0, 0): (19,) + ux.shape."""
    return torch.stack([w * (1.0 + 3.0 * c[0] * ux + (4.5 * c[0] * c[0] - 1.5) * ux * ux) for c, w in zip(_C, _W)])


class _Exact:
    """Algorithm 1 of the paper in float64: arrays indexed [z, y, x], PDFs stored less their weights."""

    def __init__(self, s, device):
        self.dev, self.s = device, s
        self.n = s['shape']
        self.per = s['periodic']
        nx, ny, nz = self.n
        t = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device=device)  # noqa: E731
        self.X, self.U, self.Om, self.R = t(s['pos']).clone(), t(s['vel']).clone(), t(s['omega']).clone(), t(s['radius'])
        self.len = t(self.n)
        self.wrap = torch.tensor([bool(p) for p in self.per], device=device)
        volume = math.pi * (2.0 * self.R) ** 3 / 6.0
        self.m = t(s['density']) * volume
        self.I = 0.4 * self.m * self.R ** 2
        g = t([0.0, 0.0, -s['gravity']])
        self.ext = (volume * (t(s['density']) - 1.0))[:, None] * g
        self.f = torch.zeros((19, nz, ny, nx), dtype=torch.float64, device=device)
        if s['flow']:
            u = s['flow'] * (torch.arange(nz, device=device, dtype=torch.float64) + 0.5) / nz
            self.f += (_equilibrium(u) - t(_W)[:, None])[:, :, None, None]
        self.body = t(s['body'])
        self.F_prev = self.T_prev = self.old = None
        self.keys = torch.zeros(0, dtype=torch.int64, device=device)
        self.spring = torch.zeros((0, 3), dtype=torch.float64, device=device)
        self.wall_spring = {}
        self.owner, self.shell = self.mapped()

    def image(self, d):
        d = torch.where(self.wrap & (d > 0.5 * self.len), d - self.len, d)
        return torch.where(self.wrap & (d < -0.5 * self.len), d + self.len, d)

    def mapped(self):
        """Owner (lowest sphere index, -1 fluid) and shell of every cell."""
        nx, ny, nz = self.n
        none = len(self.R)
        owner = torch.full((nx * ny * nz,), none, dtype=torch.int64, device=self.dev)
        shell = torch.zeros(nx * ny * nz, dtype=torch.bool, device=self.dev)
        k = int(math.ceil(float(self.R.max()) + 2.0)) + 1
        o = torch.arange(-k, k + 1, device=self.dev)
        o = torch.stack(torch.meshgrid(o, o, o, indexing='ij'), -1).reshape(-1, 3)
        cells = torch.tensor(self.n, device=self.dev)
        for a in range(0, none, 512):
            x, r = self.X[a:a + 512, None, :], self.R[a:a + 512, None]
            at = x.floor().long() + o
            d = (at + 0.5) - x
            keep = (self.wrap | ((at >= 0) & (at < cells))).all(-1)
            at = at % cells
            at = (at[..., 2] * ny + at[..., 1]) * nx + at[..., 0]
            d2 = (d * d).sum(-1)
            inside = keep & (d2 <= r * r)
            who = torch.arange(a, a + len(x), device=self.dev)[:, None].expand_as(at)
            owner.scatter_reduce_(0, at[inside], who[inside], 'amin')
            shell[at[keep & (d2 > r * r) & (d2 <= (r + 2.0) ** 2)]] = True
        owner = torch.where(owner == none, -1, owner).reshape(nz, ny, nx)
        return owner, shell.reshape(nz, ny, nx) & (owner < 0)

    def moved(self, at, c):
        """Cells at + c with periodic wrap, and which of them lie behind a wall."""
        to = at + torch.tensor(c, device=self.dev)
        cells = torch.tensor(self.n, device=self.dev)
        out = (~self.wrap & ((to < 0) | (to >= cells))).any(-1)
        return to % cells, out

    @staticmethod
    def at(v, i):
        return v[i[..., 2], i[..., 1], i[..., 0]]

    def fraction(self, r, c, R):
        a = float((c * c).sum())
        b = 2.0 * (r @ c)
        disc = b * b - 4.0 * a * ((r * r).sum(-1) - R * R)
        t = (-b - disc.clamp(min=0.0).sqrt()) / (2.0 * a)
        return torch.where(disc < 0.0, torch.full_like(t, 0.5), t).clamp(0.0, 1.0)

    def streamed(self):
        """PDFs after boundary conditions and streaming; force and torque on every sphere."""
        N = len(self.R)
        F = torch.zeros((N, 3), dtype=torch.float64, device=self.dev)
        T = torch.zeros_like(F)
        fluid = self.owner < 0
        post = torch.empty_like(self.f)
        xyz = [torch.arange(n, device=self.dev).reshape([-1 if d == a else 1 for d in (2, 1, 0)])
               for a, n in enumerate(self.n)]
        for q, c in enumerate(_C):
            p, w = _OPP[q], _W[q]
            shift = (c[2], c[1], c[0])
            val = torch.roll(self.f[q], shift, (0, 1, 2))
            out = torch.zeros_like(fluid)
            for a in (2, 1, 0):
                if self.per[a] or not c[a]:
                    continue
                up = xyz[a] - c[a]
                for side, o in enumerate((up < 0, up >= self.n[a])):
                    o = o & ~out
                    uc = -c[0] * self.s['top'] if (a, side) == (2, 1) else 0.0
                    val = torch.where(o, self.f[p] - 6.0 * w * uc, val)
                    out |= o
            src = torch.roll(self.owner, shift, (0, 1, 2))
            z, y, x = torch.nonzero(fluid & ~out & (src >= 0), as_tuple=True)
            if len(z):
                cell = torch.stack([x, y, z], -1)
                i = src[z, y, x]
                cp = -torch.tensor(c, dtype=torch.float64, device=self.dev)
                r0 = self.image((cell + 0.5) - self.X[i])
                delta = self.fraction(r0, cp, self.R[i])
                down, wall = self.moved(cell, c)
                cli = ~wall & (self.at(self.owner, down) < 0)
                r = self.image((cell + 0.5) + delta[:, None] * cp - self.X[i])
                ub = self.U[i] + torch.linalg.cross(self.Om[i], r)
                dbc = torch.where(cli, delta, torch.full_like(delta, 0.5))
                kappa = (1.0 - 2.0 * dbc) / (1.0 + 2.0 * dbc)
                fdown = torch.where(cli, self.at(self.f[p], down), torch.zeros_like(delta))
                fout, fin = self.f[p][z, y, x], self.f[q][z, y, x]
                v = fout + kappa * (fdown - fin) - 12.0 * w / (1.0 + 2.0 * dbc) * (ub @ cp)
                val[z, y, x] = v
                Fl = cp * (2.0 * w + fout + v)[:, None] - ub * (fout - v)[:, None]
                F.index_add_(0, i, Fl)
                T.index_add_(0, i, torch.linalg.cross(r, Fl))
            post[q] = val
        # links into a sphere from cells of another body count as at rest
        z, y, x = torch.nonzero(~fluid, as_tuple=True)
        solid = torch.stack([x, y, z], -1)
        own = self.owner[z, y, x]
        for q, c in enumerate(_C[1:], 1):
            to, out = self.moved(solid, [-v for v in c])
            o = self.at(self.owner, to)
            k = torch.nonzero(out | ((o >= 0) & (o != own)))[:, 0]
            i = own[k]
            cf = torch.tensor(c, dtype=torch.float64, device=self.dev)
            xc = solid[k] - cf + 0.5
            r0 = self.image(xc - self.X[i])
            far = (r0 * r0).sum(-1) > self.R[i] ** 2
            i, xc, r0 = i[far], xc[far], r0[far]
            r = self.image(xc + self.fraction(r0, cf, self.R[i])[:, None] * cf - self.X[i])
            Fl = (2.0 * _W[q] * cf).expand_as(r)
            F.index_add_(0, i, Fl)
            T.index_add_(0, i, torch.linalg.cross(r, Fl))
        return post, F, T

    def collide(self, post, a):
        """TRT with Guo forcing: even and odd parts of each pair of directions;
        the two bulk moments with their own rate in the shell."""
        tau = self.s['tau']
        sp = 1.0 / tau
        sm = 1.0 / (0.5 + 3.0 / 16.0 / (tau - 0.5))
        sb = 1.0 / (0.5 + 100.0 * (tau - 0.5))
        rho = post.sum(0)
        j = [sum(c[d] * post[q] for q, c in enumerate(_C) if c[d]) + 0.5 * float(a[d]) for d in range(3)]
        uu = j[0] ** 2 + j[1] ** 2 + j[2] ** 2
        ua = sum(j[d] * float(a[d]) for d in range(3))
        diag = sum(post[q] for q, c in enumerate(_C) if sum(v * v for v in c) == 2)
        axis = sum(post[q] for q, c in enumerate(_C) if sum(v * v for v in c) == 1)
        ds = (sb - sp) * self.shell.double()
        # change of the moments (c^2 - 1) and (1, -2, 1) of |c|^2 = 0, 1, 2 beyond rate sp
        d4 = ds * (uu - (diag - post[0]) - ua)
        d5 = -ds * (post[0] - 2.0 * axis + diag)
        new = torch.empty_like(post)
        for q, c in enumerate(_C):
            p, w, cc = _OPP[q], _W[q], sum(v * v for v in c)
            cu = sum(c[d] * j[d] for d in range(3)) + torch.zeros_like(rho)
            ca = sum(c[d] * float(a[d]) for d in range(3))
            even, odd = 0.5 * (post[q] + post[p]), 0.5 * (post[q] - post[p])
            eq = w * (rho + 4.5 * cu * cu - 1.5 * uu)
            bulk = w * (1.5 * (cc - 1.0) * d4 + 0.5 * (1.0, -2.0, 1.0)[cc] * d5)
            new[q] = (post[q] - sp * (even - eq) - sm * (odd - 3.0 * w * cu) + bulk
                      + (1.0 - 0.5 * sp) * w * (9.0 * cu * ca - 3.0 * ua) + (1.0 - 0.5 * sm) * 3.0 * w * ca)
        return new

    # -------------------------------------------------- particles

    def pairs(self):
        """Pairs i < j that may interact during a step."""
        n, found = len(self.R), []
        for a in range(0, n, 1024):
            d = self.image(self.X[a:a + 1024, None, :] - self.X[None])
            reach = self.R[a:a + 1024, None] + self.R[None] + 2.0 / 3.0 + 1.0
            i, j = torch.nonzero((d * d).sum(-1) < reach * reach, as_tuple=True)
            keep = i + a < j
            found.append(torch.stack([i[keep] + a, j[keep]]))
        self.i, self.j = torch.cat(found, 1)
        keys = self.i * n + self.j
        spring = torch.zeros((len(keys), 3), dtype=torch.float64, device=self.dev)
        if len(self.keys) and len(keys):
            k = torch.searchsorted(self.keys, keys).clamp(max=len(self.keys) - 1)
            spring = torch.where((self.keys[k] == keys)[:, None], self.spring[k], spring)
        self.keys, self.spring = keys, spring

    def lubrication(self, Ri, kr, coef, delta, n, u, om_ft, om_tt, dmin):
        mu = (self.s['tau'] - 0.5) / 3.0
        c_n, c_ftt, c_ttt, c_ftr, c_ttr = coef
        dl = torch.maximum(delta, dmin)
        on, ont = (delta > 0.0) & (delta < 2.0 / 3.0), (delta > 0.0) & (delta < 0.5)
        un = (u * n).sum(-1, keepdim=True) * n
        lg = torch.where(ont, torch.log(dl / 0.5), torch.zeros_like(dl))
        v = lambda s: s[:, None]  # noqa: E731
        pm = math.pi * mu
        F = v(torch.where(on, -6.0 * pm * Ri ** 2 * c_n * (1.0 / dl - 1.5), torch.zeros_like(dl))) * un
        F = F + v(6.0 * pm * Ri * c_ftt * lg) * (u - un)
        F = F - v(6.0 * pm * Ri ** 2 * c_ftr * lg) * torch.linalg.cross(om_ft, n)
        T = v(8.0 * pm * Ri ** 2 * c_ttt * lg) * torch.linalg.cross(u, n)
        T = T + v(8.0 * pm * Ri ** 3 * c_ttr * lg) * (om_tt - (om_tt * n).sum(-1, keepdim=True) * n)
        return F, T

    def contact(self, n, delta, ucp, u, m_eff, D, old, dt):
        """Normal and tangential contact force and the new tangential spring."""
        le, Tc = math.log(0.97), 2.31 * D * math.sqrt(3.0)
        kn, dn = m_eff * (math.pi ** 2 + le * le) / Tc ** 2, -2.0 * m_eff * le / Tc
        kappa = 2.0 * (1.0 - 0.23) / (2.0 - 0.23)
        kt, dtg = (kappa * kn)[:, None], (math.sqrt(kappa) * dn)[:, None]
        un = (u * n).sum(-1, keepdim=True) * n
        ut = ucp - un
        Fn = (-kn * delta)[:, None] * n - dn[:, None] * un
        proj = old - (old * n).sum(-1, keepdim=True) * n
        lp = proj.norm(dim=-1, keepdim=True)
        rot = torch.where(lp > 0.0, old.norm(dim=-1, keepdim=True) / lp.clamp(min=1e-300) * proj, torch.zeros_like(proj))
        Fsd = -kt * rot - dtg * ut
        fc, ls = 0.15 * Fn.norm(dim=-1, keepdim=True), Fsd.norm(dim=-1, keepdim=True)
        slip = torch.where(ls > 0.0, fc / ls.clamp(min=1e-300) * Fsd, torch.zeros_like(Fsd))
        stick = ls < fc
        return Fn, torch.where(stick, Fsd, slip), torch.where(stick, rot + dt * ut, -(slip + dtg * ut) / kt)

    def forces(self, Fbar, Tbar, dt, keep):
        F, T = Fbar + self.ext, Tbar.clone()
        cross = torch.linalg.cross
        i, j = self.i, self.j
        if len(i):
            d = self.image(self.X[i] - self.X[j])
            dist = d.norm(dim=-1)
            n = d / dist[:, None]
            delta = dist - (self.R[i] + self.R[j])
            u = self.U[i] - self.U[j]
            Rm = 0.5 * (self.R[i] + self.R[j])
            dmin = (0.001 + 0.00007 * Rm) * Rm
            for a, b, s in ((i, j, 1.0), (j, i, -1.0)):
                Ri, k = self.R[a], self.R[b] / self.R[a]
                coef = (k * k / (1 + k) ** 2, 4 * k * (2 + k + 2 * k * k) / (15 * (1 + k) ** 3),
                        k * (4 + k) / (10 * (1 + k) ** 2), 2 * k * k / (15 * (1 + k) ** 2), 2 * k / (5 * (1 + k)))
                oi, oj, kk = self.Om[a], self.Om[b], k[:, None]
                Fl, Tl = self.lubrication(Ri, k, coef, delta, s * n, s * u, oi + oj + 4 / kk * oi + 4 * kk * oj,
                                          oi + kk / 4 * oj, dmin)
                F.index_add_(0, a, Fl)
                T.index_add_(0, a, Tl)
            ri, rj = -0.5 * d, 0.5 * d
            ucp = (self.U[i] + cross(self.Om[i], ri)) - (self.U[j] + cross(self.Om[j], rj))
            m_eff = self.m[i] * self.m[j] / (self.m[i] + self.m[j])
            Fn, Ft, new = self.contact(n, delta, ucp, u, m_eff, self.R[i] + self.R[j], self.spring, dt)
            hit = (delta < 0.0)[:, None]
            Fc, Ft = torch.where(hit, Fn + Ft, 0.0), torch.where(hit, Ft, 0.0)
            F.index_add_(0, i, Fc)
            F.index_add_(0, j, -Fc)
            T.index_add_(0, i, cross(ri, Ft))
            T.index_add_(0, j, cross(rj, -Ft))
            if keep:
                self.spring = torch.where(hit, new, 0.0)
        one = torch.ones_like(self.R)
        for a in range(3):
            for side in range(2) if not self.per[a] else ():
                n = torch.zeros_like(self.X)
                n[:, a] = 1.0 - 2.0 * side
                delta = (self.X[:, a] - side * self.n[a]) * (1.0 - 2.0 * side) - self.R
                u = self.U.clone()
                if (a, side) == (2, 1):
                    u[:, 0] -= self.s['top']
                coef = (one, 8 / 15 * one, one / 10, 2 / 15 * one, 2 / 5 * one)
                Fl, Tl = self.lubrication(self.R, None, coef, delta, n, u, self.Om, self.Om,
                                          (0.001 + 0.00007 * self.R) * self.R)
                ri = -(self.R + 0.5 * delta)[:, None] * n
                old = self.wall_spring.get((a, side), torch.zeros_like(self.X))
                Fn, Ft, new = self.contact(n, delta, u + cross(self.Om, ri), u, self.m, 2.0 * self.R, old, dt)
                hit = (delta < 0.0)[:, None]
                F = F + Fl + torch.where(hit, Fn + Ft, 0.0)
                T = T + Tl + torch.where(hit, cross(ri, Ft), 0.0)
                if keep:
                    self.wall_spring[a, side] = torch.where(hit, new, 0.0)
        return F, T

    def wrapped(self, X):
        X = torch.where(self.wrap & (X >= self.len), X - self.len, X)
        return torch.where(self.wrap & (X < 0.0), X + self.len, X)

    def refill(self, before, a):
        """PDFs of cells that a sphere has left, from their fluid neighbours."""
        z, y, x = torch.nonzero((before >= 0) & (self.owner < 0), as_tuple=True)
        if not len(z):
            return
        cell = torch.stack([x, y, z], -1)
        i = before[z, y, x]
        ok, drho, vel = [], [], []
        for c in _C:
            to, out = self.moved(cell, c)
            ok.append(~out & (self.at(before, to) < 0) & (self.at(self.owner, to) < 0))
            f = self.f[:, to[:, 2], to[:, 1], to[:, 0]]
            drho.append(f.sum(0))
            vel.append(torch.stack([sum(e[d] * f[q] for q, e in enumerate(_C) if e[d]) - 0.5 * a[d] for d in range(3)], -1))
        count = sum(o.double() for o in ok[1:])
        total = sum(torch.where(o, r, 0.0) for o, r in zip(ok[1:], drho[1:]))
        dr = torch.where(count > 0, total / count.clamp(min=1.0), 0.0)
        rho = 1.0 + dr
        ut = self.U[i] + torch.linalg.cross(self.Om[i], self.image((cell + 0.5) - self.X[i]))
        grad = []
        for e in ((1, 0, 0), (0, 1, 0), (0, 0, 1)):
            p, m = _C.index(e), _C.index(tuple(-v for v in e))
            op, om = ok[p][:, None], ok[m][:, None]
            grad.append(torch.where(op & om, 0.5 * (vel[p] - vel[m]),
                                    torch.where(op, vel[p] - ut, torch.where(om, ut - vel[m], 0.0))))
        g = torch.stack(grad, -1)
        P = rho[:, None, None] * (ut[:, :, None] * ut[:, None, :] - self.s['tau'] / 3.0 * (g + g.transpose(1, 2)))
        trace = P.diagonal(dim1=1, dim2=2).sum(-1) / 3.0
        for q, c in enumerate(_C):
            cf = torch.tensor(c, dtype=torch.float64, device=self.dev)
            self.f[q, z, y, x] = _W[q] * (dr + 3.0 * rho * (ut @ cf) + 4.5 * ((P @ cf) @ cf - trace))

    def step(self):
        a = self.body
        if self.s['counter']:
            a = a - self.ext.sum(0) / float((self.owner < 0).sum())
        self.a = a
        dem = self.s['motion'] == L.MOTION_DEM
        if dem:
            self.pairs()
            if self.F_prev is None:
                zero = torch.zeros_like(self.X)
                self.F_prev, self.T_prev = self.forces(zero, zero, 0.0, False)
        post, F, T = self.streamed()
        old = self.old or (F, T)
        Fbar, Tbar = 0.5 * (F + old[0]), 0.5 * (T + old[1])
        self.old = (F, T)
        self.f = self.collide(post, a)
        del post
        if self.s['motion'] == L.MOTION_FIXED:
            return
        if dem:
            dt, m, I = 0.1, self.m[:, None], self.I[:, None]
            for _ in range(10):
                self.X = self.wrapped(self.X + dt * self.U + dt * dt / (2.0 * m) * self.F_prev)
                Fn, Tn = self.forces(Fbar, Tbar, dt, True)
                self.U = self.U + dt / (2.0 * m) * (self.F_prev + Fn)
                self.Om = self.Om + dt / (2.0 * I) * (self.T_prev + Tn)
                self.F_prev, self.T_prev = Fn, Tn
        else:
            self.X = self.wrapped(self.X + self.U)
        before = self.owner
        self.owner, self.shell = self.mapped()
        self.refill(before, a)

    def density(self, points):
        """Trilinear density at points, solid cells counting 1."""
        rho = 1.0 + torch.where(self.owner < 0, self.f.sum(0), 0.0)
        g = torch.as_tensor(points, device=self.dev) - 0.5
        base = g.floor()
        got = 0.0
        for c in range(8):
            o = torch.tensor([(c >> d) & 1 for d in range(3)], device=self.dev)
            w = torch.where(o > 0, g - base, 1.0 - (g - base)).prod(-1)
            cells = torch.tensor(self.n, device=self.dev)
            i = base.long() + o
            i = torch.where(self.wrap, i % cells, torch.minimum(i.clamp(min=0), cells - 1))
            got = got + w * self.at(rho, i)
        return got.cpu().numpy()

    def outputs(self, fields):
        out = dict(pos=self.X, vel=self.U, omega=self.Om, force_hyd=self.old[0], torque_hyd=self.old[1])
        if fields:
            fluid = self.owner < 0
            out['rho'] = torch.where(fluid, 1.0 + self.f.sum(0), 0.0)
            out['u'] = torch.stack([torch.where(fluid, sum(c[d] * self.f[q] for q, c in enumerate(_C) if c[d])
                                                - 0.5 * self.a[d], 0.0) for d in range(3)])
            out['flags'] = None
        return {k: v if v is None else v.cpu().numpy() for k, v in out.items()}


def exact(case, seed):
    if case['kind'] == 'map':
        return None     # whole numbers
    device = 'cuda' if torch.cuda.is_available() else 'cpu'
    if case['kind'] == 'batch':
        got = []
        for s in _boxes(case, seed):
            e = _Exact(s, device)
            for _ in range(1 + case['steps']):
                e.step()
            got.append(e.outputs(False))
        return {k: np.concatenate([g[k] for g in got]) for k in got[0]}
    s = _setup(case, seed)
    e = _Exact(s, device)
    if case['kind'] == 'probe':
        rho, x = [], s['pos'][0].copy()
        for k in range(case['steps']):
            vel, omega = _fall(s, k + 1)
            e.U, e.Om = torch.as_tensor(vel, device=device), torch.as_tensor(omega, device=device)
            e.step()
            x = (x + vel[0]) % s['shape'][2]
            rho.append(e.density(_probe_points(case, s, x)))
        return dict(rho=np.array(rho), **e.outputs(False))
    for _ in range(case['steps']):
        e.step()
    cells = case['nx'] * case['ny'] * case['nz']
    return e.outputs(cells <= FIELDS_MAX and case['kind'] != 'shear')
