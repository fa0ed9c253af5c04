"""What a user of this framework has it do, as timed cases.

Every case goes through the package's public entry points
(``binding.Simulation``, ``binding.Server``, ``ibm_lbm_spread_noalloc``): a
program makes a handle once, advances it, and reads the result back. Families:

* ``tube``    red-cell membranes in a body-force-driven tube (blood flow);
* ``channel`` red cells and filaments with Morse excluded volume between walls;
* ``shear``   one rigid ellipsoid in a Couette cell (Jeffery orbits);
* ``serve``   a batch of independent shear cells through the server;
* ``tracers`` passive tracers carried by a flow without bodies;
* ``stretch`` solid-only stretching of red cells (no fluid);
* ``spread``  force spreading without a handle, on device arrays.

Results come as a program stores them in a trajectory file: whole arrays, in
single precision. The library computes velocities, densities and forces in
FP32 and its C ABI carries them in FP64 arrays. Cells start deformed (a few
per cent of strain), as they are in a flow.
"""
import functools
import math

import numpy as np
import torch

from paper_1704_04551_gb300 import binding, inputs

STORAGE_BYTES = {'f32': 4, 'f16': 2, 'bf16': 2}
DIAMETER = 16.0     # red cells: 8 um at dx = 0.5 um


def listed():
    return [
        # a framework's own time loop spreads the forces of one small body per call
        dict(name='spread_body', kind='spread', nx=48, ny=40, nz=36, geometry=1, markers=812, clustered=True),
        # the same entry point near its largest lattice, markers all over it
        dict(name='spread_dense', kind='spread', nx=101, ny=97, nz=103, geometry=0, markers=120000, clustered=False),
        # the 500-step Jeffery validation cell
        dict(name='shear_32', kind='shear', nx=32, ny=32, nz=32, freq=9, direct=False, steps=500),
        # a monitored run: a few steps, then the pose, the markers and the fields
        dict(name='shear_monitor', kind='shear', nx=60, ny=47, nz=33, freq=9, direct=True, steps=10),
        # continuous batching of independent shear cells of mixed sizes
        dict(name='serve_24', kind='serve', cases=24, L_min=24, L_max=96, steps=800, slots=16, chunk=100),
        # optical-tweezer stretching of one fine cell
        dict(name='stretch_1442', kind='stretch', freq=12, bodies=1, steps=500),
        # tracers scattered through a periodic flow
        dict(name='tracers_box', kind='tracers', nx=131, ny=96, nz=110, geometry=0, markers=150000, storage='f32',
             steps=50),
        # 64^3 copy of the tube with 50 cells
        dict(name='tube_64', kind='tube', nx=64, ny=64, radius=30.0, cells=50, tumbling=False, storage='f32',
             steps=200),
        # dilute tube, cells at any orientation (tumbling), BF16 storage, ragged sizes
        dict(name='tube_tumbling', kind='tube', nx=203, ny=118, radius=56.0, cells=170, tumbling=True,
             storage='bf16', steps=100),
        # the headline tube: 256^3, 3000 cells
        dict(name='tube_256', kind='tube', nx=256, ny=256, radius=120.0, cells=3000, tumbling=False, storage='f32',
             steps=200),
        # the same with populations stored in half precision
        dict(name='tube_256_f16', kind='tube', nx=256, ny=256, radius=120.0, cells=3000, tumbling=False,
             storage='f16', steps=200),
        # the large mixed suspension: 512^3, 20000 cells, 4000 filaments, trajectory output
        dict(name='channel_512', kind='channel', nx=512, ny=512, nz=512, cells=20000, filaments=4000, storage='f16',
             steps=50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def draw(rng):
    kind = rng.choice(['spread', 'shear', 'serve', 'tracers', 'stretch', 'tube', 'tube', 'channel'])
    if kind == 'spread':
        n = [_log(rng, 16, 100) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], geometry=rng.randrange(3), markers=_log(rng, 100, 120000),
                    clustered=rng.random() < 0.5)
    if kind == 'shear':
        n = [_log(rng, 24, 96) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], freq=rng.randint(7, 9), direct=rng.random() < 0.4,
                    steps=_log(rng, 1, 500))
    if kind == 'serve':
        return dict(kind=kind, cases=rng.randint(4, 24), L_min=24, L_max=rng.randint(32, 96),
                    steps=_log(rng, 200, 800), slots=rng.choice([8, 16, 32]), chunk=rng.choice([50, 100]))
    if kind == 'tracers':
        n = [_log(rng, 24, 160) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], geometry=rng.randrange(3), markers=_log(rng, 500, 300000),
                    storage=rng.choice(['f32', 'f16', 'bf16']), steps=_log(rng, 10, 100))
    if kind == 'stretch':
        return dict(kind=kind, freq=rng.randint(5, 16), bodies=_log(rng, 1, 64), steps=_log(rng, 50, 500))
    if kind == 'tube':
        ny = _log(rng, 40, 200)
        nx = _log(rng, 40, 256)
        radius = round(ny / 2.0 - rng.uniform(2.0, 4.0), 1)
        tumbling = rng.random() < 0.4
        most = len(_tube_slots(nx, ny, radius, tumbling)[0])
        return dict(kind=kind, nx=nx, ny=ny, radius=radius, cells=max(1, int(most * rng.uniform(0.3, 0.9))),
                    tumbling=tumbling, storage=rng.choice(['f32', 'f16', 'bf16']), steps=_log(rng, 18, 200))
    n = [_log(rng, 96, 256), _log(rng, 48, 256), _log(rng, 48, 256)]
    most = len(_channel_slots(*n)[0])
    sites = len(_filament_sites(n[1], n[2]))
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], cells=max(1, int(most * rng.uniform(0.2, 0.6))),
                filaments=max(1, int(sites * rng.uniform(0.05, 0.3))), storage=rng.choice(['f32', 'f16', 'bf16']),
                steps=_log(rng, 10, 50))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _sphere(freq):
    return inputs.geodesic_sphere(freq)


@functools.lru_cache(maxsize=None)
def _red_cell(freq):
    return inputs.rbc_rest_shape(DIAMETER, freq)


def _rotations(q):
    """Rotation matrices [n][3][3] of unit quaternions [n][4]."""
    w, x, y, z = q.T
    R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                  [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                  [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])
    return np.moveaxis(R, 2, 0)


def _random_rotations(rng, n):
    q = rng.standard_normal((n, 4))
    return _rotations(q / np.linalg.norm(q, axis=1, keepdims=True))


def _stacked_rotations(rng, tilt):
    """Cells whose axis lies along x, spun about it and tilted by `tilt` (radians, [n])."""
    n = len(tilt)
    spin, az = 2 * np.pi * rng.random((2, n))
    zero = np.zeros(n)
    align = np.tile([[0.0, 0, 1], [0, 1, 0], [-1, 0, 0]], (n, 1, 1))    # body z -> x
    own = _rotations(np.stack([np.cos(spin / 2), zero, zero, np.sin(spin / 2)], 1))
    t = _rotations(np.stack([np.cos(tilt / 2), zero, np.sin(tilt / 2) * np.cos(az), np.sin(tilt / 2) * np.sin(az)], 1))
    return t @ align @ own


def _hex_columns(reach, spacing):
    m = int(reach // spacing) + 2
    i, j = np.meshgrid(np.arange(-m, m + 1), np.arange(-m, m + 1), indexing='ij')
    return np.stack([spacing * (i + 0.5 * j).ravel(), spacing * (j * math.sqrt(3) / 2).ravel()], 1)


def _slots(x0, x1, columns, pitch):
    per = max(1, int((x1 - x0) // pitch))
    x = x0 + (np.arange(per) + 0.5) * (x1 - x0) / per
    P = np.concatenate([np.repeat(x[None], len(columns), 0).reshape(-1, 1), np.repeat(columns, per, 0)], 1)
    return P, per


def _tube_slots(nx, ny, radius, tumbling):
    """Places for cells in a tube: stacks of discs, or room for any orientation."""
    spacing = DIAMETER + 2.0
    cols = _hex_columns(radius, spacing)
    cols = cols[(cols ** 2).sum(1) <= (radius - DIAMETER / 2 - 1.0) ** 2] + (ny - 1) / 2.0
    return _slots(0.0, nx, cols, spacing if tumbling else 6.53)


def _channel_slots(nx, ny, nz):
    y = np.arange(9.5, ny - 10.0, DIAMETER + 2.0)
    z = np.arange(9.5, nz - 10.0, DIAMETER + 2.0)
    cols = np.stack(np.meshgrid(y, z, indexing='ij'), -1).reshape(-1, 2)
    return _slots(53.0, nx - 1.0, cols, 6.53)


def _filament_sites(ny, nz):
    y, z = np.arange(1.5, ny - 1.5, 3.0), np.arange(0.5, nz - 0.5, 3.0)
    return np.stack(np.meshgrid(y, z, indexing='ij'), -1).reshape(-1, 2)


def _cells(rng, slots, per, n, tumbling):
    """n red cells in a random subset of the slots: positions [3][n V], bodies."""
    rest, tris = _red_cell(8)
    V = rest.shape[1]
    pick = np.sort(rng.permutation(len(slots))[:n])
    c = slots[pick] + rng.uniform(-0.25, 0.25, (n, 3))
    if tumbling:
        R = _random_rotations(rng, n)
    else:
        # room to tilt depends on the neighbouring places of the stack
        full = np.zeros(len(slots), bool)
        full[pick] = True
        full = full.reshape(-1, per)
        near = (np.roll(full, 1, 1).astype(int) + np.roll(full, -1, 1)).ravel()[pick]
        R = _stacked_rotations(rng, np.radians(np.array([40.0, 20.0, 6.0])[near]) * np.sqrt(rng.random(n)))
    strain = np.exp(rng.uniform(-0.06, 0.06, (n, 3)))
    X = np.einsum('bij,bjv->ibv', R * strain[:, None, :], np.broadcast_to(rest, (n, 3, V)))
    X += c.T[:, :, None]
    mod = inputs.rbc_moduli_lattice(0.5e-6, 1.0)
    keys = ('kBT_p', 'k_b', 'k_l', 'k_g', 'k_v')
    s = 1.0 + 0.2 * rng.uniform(-1, 1, (n, 5))
    bodies = [dict(kind=0, first=b * V, count=V, **{k: mod[k] * s[b, j] for j, k in enumerate(keys)}) for b in range(n)]
    return np.ascontiguousarray(X.reshape(3, -1)), bodies, dict(rest_X=rest, tris=tris)


def _tube(c, seed):
    rng = np.random.default_rng(seed)
    slots, per = _tube_slots(c['nx'], c['ny'], c['radius'], c['tumbling'])
    X, bodies, mesh = _cells(rng, slots, per, c['cells'], c['tumbling'])
    nu, R = 1.0 / 6.0, c['radius']
    g = 4.0 * nu * (nu / (2.0 * R)) / (R * R)     # centreline Reynolds number 1
    lat = dict(nx=c['nx'], ny=c['ny'], nz=c['ny'], tau=1.0, geometry=2, tube_radius=R, body_force=[g, 0.0, 0.0])
    return dict(lattice=lat, mesh=mesh, bodies=bodies, X=X)


def _channel(c, seed):
    rng = np.random.default_rng(seed)
    nx, ny, nz = c['nx'], c['ny'], c['nz']
    slots, per = _channel_slots(nx, ny, nz)
    X, bodies, mesh = _cells(rng, slots, per, c['cells'], False)
    n, beads = c['filaments'], 50
    sites = _filament_sites(ny, nz)
    at = sites[np.sort(rng.permutation(len(sites))[:n])] + rng.uniform(-0.2, 0.2, (n, 2))
    F = np.empty((3, n, beads))
    F[0] = 1.0 + 0.5 * rng.random((n, 1)) + np.arange(beads)
    # slightly bent chains
    phase, amp = 2 * np.pi * rng.random((n, 1)), 0.25 * rng.random((n, 1))
    F[1] = at[:, :1] + amp * np.sin(0.2 * np.arange(beads) + phase)
    F[2] = at[:, 1:] + amp * np.cos(0.2 * np.arange(beads) + phase)
    soft, stiff = (inputs.filament_moduli_lattice(0.5e-6, 1.0, k) for k in (4.1e-20, 4.1e-18))
    first = X.shape[1]
    bodies += [dict(kind=2, first=first + k * beads, count=beads, l0=1.0, **(stiff if k & 1 else soft))
               for k in range(n)]
    u = inputs.lattice_units(0.5e-6, 1.0)
    g = 2.0 / 6.0 * (1000.0 * u['dt']) / ny       # wall shear rate 1000 1/s
    lat = dict(nx=nx, ny=ny, nz=nz, tau=1.0, geometry=1, wall_u=[0.0, 0.0], body_force=[g, 0.0, 0.0])
    return dict(lattice=lat, mesh=mesh, bodies=bodies, X=np.concatenate([X, F.reshape(3, -1)], 1),
                morse=inputs.morse_lattice(0.5e-6, 1.0))


def _couette(nx, ny, nz, gamma, rng, freq, direct):
    """One neutrally buoyant ellipsoid in a wall-driven shear cell that has reached its linear profile."""
    L = min(nx, ny, nz)
    a = 0.1875 * L
    # direct forcing is explicit: it takes bodies with some mass behind their surface
    b = a / rng.uniform(1.1, 1.5) if direct else max(a / rng.uniform(1.5, 5.0), 1.5)
    q = rng.standard_normal(4)
    q /= np.linalg.norm(q)
    S = _sphere(freq)[0]
    C = np.array([(nx - 1) / 2, (ny - 1) / 2, (nz - 1) / 2]) + rng.uniform(-0.5, 0.5, 3)
    X = (_rotations(q[None])[0] @ (S * [a, b, b]).T) + C[:, None]
    area, ref = inputs.ellipsoid_area(a, b, b), inputs.ellipsoid_area(6.0, 3.0, 3.0)
    mass = 4 / 3 * math.pi * a * b * b
    body = dict(kind=3 if direct else 1, first=0, count=X.shape[1], mass=mass,
                kappa=area / X.shape[1] if direct else 0.02 * area / ref * 812 / X.shape[1],
                inertia=[mass * 2 * b * b / 5, mass * (a * a + b * b) / 5, mass * (a * a + b * b) / 5],
                center=C.tolist(), quat=q.tolist(), vel=[0.0] * 3, omega=[0.0, 0.0, -0.5 * gamma])
    wall = 0.5 * gamma * ny
    y = np.arange(ny)
    u0 = np.zeros((3, nz, ny, nx))
    u0[0] = (wall * (2.0 * (y + 0.5) / ny - 1.0))[None, :, None]
    lat = dict(nx=nx, ny=ny, nz=nz, tau=0.8, geometry=1, wall_u=[-wall, wall], body_force=[0.0, 0.0, 0.0])
    return dict(lattice=lat, mesh=None, bodies=[body], X=np.ascontiguousarray(X), u0=u0.reshape(3, -1))


def _shear(c, seed):
    rng = np.random.default_rng(seed)
    return _couette(c['nx'], c['ny'], c['nz'], math.exp(rng.uniform(math.log(2e-4), math.log(1e-3))), rng, c['freq'],
                    c['direct'])


def _served(c, seed):
    rng = np.random.default_rng(seed)
    # the sizes fill the range evenly, so that one batch's work does not depend on the seed
    sizes = np.linspace(c['L_min'], c['L_max'], c['cases']).astype(int)
    out = []
    for L in rng.permutation(sizes):
        gamma = math.exp(rng.uniform(math.log(1e-4), math.log(1e-3)))
        out.append(_couette(int(L), int(L), int(L), gamma, rng, 9, False))
    return out


def _tracers(c, seed):
    rng = np.random.default_rng(seed)
    nx, ny, nz = c['nx'], c['ny'], c['nz']
    R = 0.5 * min(ny, nz) - 1.5
    lat = dict(nx=nx, ny=ny, nz=nz, tau=0.7, geometry=c['geometry'], tube_radius=R if c['geometry'] == 2 else 0.0,
               wall_u=[-0.01, 0.01], body_force=[2e-6, 0.0, 0.0])
    M = c['markers']
    if c['geometry'] == 2:
        r, th = (R - 1.0) * np.sqrt(rng.random(M)), 2 * np.pi * rng.random(M)
        X = np.stack([nx * rng.random(M), (ny - 1) / 2 + r * np.cos(th), (nz - 1) / 2 + r * np.sin(th)])
    else:
        X = rng.random((3, M)) * np.array([[nx], [ny - 1.0], [nz]])
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing='ij', sparse=True)
    kx, ky, kz = (2 * np.pi / n for n in (nx, ny, nz))
    p = 2 * np.pi * rng.random(3)
    u0 = 0.02 * np.stack([np.sin(kx * x + p[0]) * np.cos(ky * y + p[1]) * np.cos(kz * z + p[2]),
                          -np.cos(kx * x + p[0]) * np.sin(ky * y + p[1]) * np.cos(kz * z + p[2]),
                          0.2 * np.cos(kx * x + p[0]) * np.sin(kz * z + p[2]) + 0.0 * y])
    return dict(lattice=lat, mesh=None, bodies=[], X=X, u0=u0.reshape(3, -1))


def _stretch(c, seed):
    rng = np.random.default_rng(seed)
    rest, tris = _red_cell(c['freq'])
    V, n = rest.shape[1], c['bodies']
    u, mod = inputs.lattice_units(0.5e-6, 1.0), inputs.rbc_moduli_lattice(0.5e-6, 1.0)
    # the mesh's own kBT/p, from the shear modulus 6 uN/m (about 1.25 sqrt(3) (kBT/p) / l0)
    l0 = math.sqrt(4 / math.sqrt(3) * 540.0 / len(tris))
    kBT_p = 6e-6 / (u['force'] / 0.5e-6) * l0 / (1.25 * math.sqrt(3.0))
    X, F, bodies = np.empty((3, n, V)), np.zeros((3, n, V)), []
    patch = max(1, int(round(0.05 * V)))
    order = np.argsort(rest[0])
    for b in range(n):
        strain = np.exp(rng.uniform(-0.04, 0.04, 3))
        X[:, b] = rest * strain[:, None] + 32.0 + 40.0 * b * np.array([[0.0], [1.0], [0.0]])
        pull = rng.uniform(10.0, 40.0) * 1e-12 / u['force'] / patch
        F[0, b, order[:patch]], F[0, b, order[-patch:]] = -pull, pull
        bodies.append(dict(kind=0, first=b * V, count=V, kBT_p=kBT_p * rng.uniform(0.8, 1.2),
                           **{k: mod[k] for k in ('k_b', 'k_l', 'k_g', 'k_v')}))
    lat = dict(nx=16, ny=16, nz=16, tau=1.0, geometry=0)
    return dict(lattice=lat, mesh=dict(rest_X=rest, tris=tris), bodies=bodies, X=X.reshape(3, -1)), F.reshape(3, -1)


def _spread(c, seed):
    rng = np.random.default_rng(seed)
    n, M = np.array([c['nx'], c['ny'], c['nz']], dtype=float)[:, None], c['markers']
    if c['clustered']:    # one body: a sphere's surface in the middle
        d = rng.standard_normal((3, M))
        X = 0.5 * (n - 1) + 0.25 * n.min() * d / np.linalg.norm(d, axis=0) + rng.uniform(-1, 1, (3, 1))
    else:
        X = rng.random((3, M)) * (n - 1)
    return X, 1e-3 * rng.standard_normal((3, M)), 0.5 * min(c['ny'], c['nz']) - 1.5


def prepare(case, seed):
    k = case['kind']
    if k == 'spread':
        X, F, R = _spread(case, seed)
        g = torch.empty(3, case['nx'] * case['ny'] * case['nz'], dtype=torch.float64, device='cuda')
        return dict(case=case, X=torch.from_numpy(X).cuda(), F=torch.from_numpy(F).cuda(), R=R, g=g)
    if k == 'serve':
        return dict(case=case, cells=_served(case, seed),
                    server=binding.Server(64 << 30, max_active=case['slots'], chunk_steps=case['chunk']))
    if k == 'stretch':
        w, F = _stretch(case, seed)
        return dict(case=case, sim=binding.Simulation.from_workload(w), F=F)
    make = dict(tube=_tube, channel=_channel, shear=_shear, tracers=_tracers)[k]
    sim = binding.Simulation.from_workload(make(case, seed), storage=case.get('storage', 'f32'))
    return dict(case=case, sim=sim)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _single(*arrays):
    # torch's threads pay for themselves from some megabytes on only
    return [torch.from_numpy(a).to(torch.float32) if a.size > 1 << 22 else torch.from_numpy(a.astype(np.float32))
            for a in arrays]


def run(state):
    case = state['case']
    k = case['kind']
    if k == 'spread':
        X, F, g = state['X'], state['F'], state['g']
        rc = binding.ibm_lbm_spread_noalloc(X.data_ptr(), F.data_ptr(), X.shape[1], case['nx'], case['ny'], case['nz'],
                                            case['geometry'], state['R'], g.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        if rc != binding.OK:
            raise RuntimeError(f'spread: {rc}')
        return g
    if k == 'serve':
        srv = state['server']
        ids = [srv.submit(w, case['steps']) for w in state['cells']]
        while True:
            rc, running, pending, _ = srv.advance()
            if rc != binding.OK:
                raise RuntimeError(f'serve: {rc}')
            if running == 0 and pending == 0:
                break
        done = [srv.result(i) for i in ids]
        join = lambda key: np.concatenate([r[key].ravel() for r in done])  # noqa: E731
        pose = np.array([b[q] for r in done for b in r['bodies'] for q in ('center', 'quat', 'vel', 'omega')
                         for b[q] in [b[q] + [0.0] * (4 - len(b[q]))]])
        return dict(zip(('rho', 'u', 'X', 'U', 'pose'), _single(*map(join, ('rho', 'u', 'X', 'U')), pose)))
    sim = state['sim']
    if k == 'stretch':
        sim.solid_steps(case['steps'], 1.0, 0.05, 1.0, state['F'])
        X, _, F = sim.markers()
        return dict(zip(('X', 'F'), _single(X, F)))
    sim.step(case['steps'])
    out = dict(zip(('X', 'U', 'F'), _single(*sim.markers())))
    if k == 'tracers':
        del out['F']      # always zero
    if k == 'shear':
        b = sim.bodies()[0]
        out['pose'] = _single(np.array(b['center'] + b['quat'] + b['vel'] + b['omega']))[0]
    if k != 'channel':    # there the trajectory is written more often than the fields
        out.update(zip(('rho', 'u'), _single(*sim.fields())))
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _fluid_cells(c):
    if c['kind'] == 'tube':
        return int(math.pi * c['radius'] ** 2 * c['nx'])
    if c.get('geometry') == 2:
        return int(math.pi * (0.5 * min(c['ny'], c['nz']) - 1.5) ** 2 * c['nx'])
    return c['nx'] * c['ny'] * c['nz']


def work(case):
    """One pass: populations read and written once a step (19 each), the force
    density read and the velocity written where stencils reach (24 bytes a
    cell), positions read and written and velocity and force handed over (72
    bytes a marker), and the results written once at the end."""
    c, k = case, case['kind']
    if k == 'spread':
        N, M = c['nx'] * c['ny'] * c['nz'], c['markers']
        return dict(bytes=48 * M + 24 * N, flops=M * 64 * 7)
    if k == 'stretch':
        V, n = 10 * c['freq'] ** 2 + 2, c['bodies']
        # positions and velocities stay on the chip between steps in principle: the floor is the arithmetic
        return dict(bytes=(48 + 24 + 24 + 48) * n * V, flops=c['steps'] * n * V * (3 * 250 + 2 * 120 + 30))
    if k == 'serve':
        Ls = np.linspace(c['L_min'], c['L_max'], c['cases']).astype(int)
        N, M = int((Ls.astype(np.int64) ** 3).sum()), 812 * c['cases']
        near, s, steps = 2000 * c['cases'], 4, c['steps']
        ends = 32 * N + 48 * M
    else:
        N = _fluid_cells(c)
        s, steps = STORAGE_BYTES[c.get('storage', 'f32')], c['steps']
        if k == 'shear':
            M, near = 10 * c['freq'] ** 2 + 2, 2000
        elif k == 'tracers':
            M = c['markers']
            near = int(N * (1 - math.exp(-64.0 * M / N)))
        else:
            M = 642 * c['cells'] + 50 * c.get('filaments', 0)
            near = 2300 * c['cells'] + 800 * c.get('filaments', 0)
        ends = 72 * M + (0 if k == 'channel' else 32 * c['nx'] * c['ny'] * c.get('nz', c['ny']))
    near = min(near, N)
    edges = 3 * 642 * c.get('cells', 0) if k in ('tube', 'channel') else 0
    return dict(bytes=steps * (38 * s * N + 24 * near + 72 * M) + ends,
                flops=steps * (250 * N + M * 64 * 13 + 330 * edges))


# ---------------------------------------------------------------------------
# the same in 64 bits, with torch alone
# ---------------------------------------------------------------------------
D3Q19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
         (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
         (0, -1, 1)]
F64 = torch.float64


def _device():
    return torch.device('cuda' if torch.cuda.is_available() else 'cpu')


class _Nodes:
    """The 4^3 stencil of every marker: node indices and weights [M][64] (weight 0 on solid nodes)."""

    def __init__(self, grid, X):
        nx, ny, nz = grid.n
        base = torch.floor(X)
        r = torch.arange(-1, 3, device=X.device, dtype=F64)[None, None] - (X - base)[:, :, None]      # [3][M][4]
        w = 0.25 * (1 + torch.cos(0.5 * math.pi * r))
        p = base[:, :, None].long() + torch.arange(-1, 3, device=X.device)[None, None]
        x, y, z = p[0] % nx, p[1], p[2]
        if grid.geometry == 0:
            y = y % ny
        if grid.geometry != 2:
            z = z % nz
        ok_y, ok_z = (y >= 0) & (y < ny), (z >= 0) & (z < nz)
        w = [w[0], w[1] * ok_y, w[2] * ok_z]
        y, z = y.clamp(0, ny - 1), z.clamp(0, nz - 1)
        M = X.shape[1]
        wzy = w[2][:, :, None] * w[1][:, None, :]
        if grid.geometry == 2:
            wzy = wzy * grid.fluid_zy[z[:, :, None], y[:, None, :]]
        self.i = (x[:, None, None, :] + nx * (y[:, None, :, None] + ny * z[:, :, None, None])).reshape(M, 64)
        self.w = (wzy[:, :, :, None] * w[0][:, None, None, :]).reshape(M, 64)


class _Grid:
    def __init__(self, lat):
        dev = _device()
        self.n = nx, ny, nz = lat['nx'], lat['ny'], lat['nz']
        self.geometry = lat['geometry']
        z, y = torch.meshgrid(torch.arange(nz, device=dev), torch.arange(ny, device=dev), indexing='ij')
        self.fluid_zy = torch.ones(nz, ny, dtype=torch.bool, device=dev)
        if self.geometry == 2:
            R2 = float(np.float32(lat['tube_radius'] ** 2))
            self.fluid_zy = (y - (ny - 1) / 2.0) ** 2 + (z - (nz - 1) / 2.0) ** 2 <= R2
        self.fluid = self.fluid_zy[:, :, None].expand(nz, ny, nx).reshape(-1)


class _Fluid(_Grid):
    """D3Q19 BGK with Guo forcing and half-way bounce-back, two arrays, gather streaming."""

    def __init__(self, lat, u0=None):
        super().__init__(lat)
        dev = _device()
        nx, ny, nz = self.n
        N = nx * ny * nz
        self.tau = lat['tau']
        self.c = torch.tensor(D3Q19, dtype=F64, device=dev)
        self.wt = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=F64, device=dev)
        self.g0 = torch.tensor(lat.get('body_force', [0.0] * 3), dtype=F64, device=dev)[:, None]
        opp = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
        x = torch.arange(nx, device=dev)[None, None, :]
        y = torch.arange(ny, device=dev)[None, :, None]
        z = torch.arange(nz, device=dev)[:, None, None]
        here = x + nx * (y + ny * z)
        self.src = torch.empty(19, N, dtype=torch.int64, device=dev)
        self.wall = []
        for i, (cx, cy, cz) in enumerate(D3Q19):
            sx, sy, sz = (x - cx) % nx, y - cy, z - cz
            solid = torch.zeros(nz, ny, 1, dtype=torch.bool, device=dev)
            if self.geometry != 0:
                solid = solid | (sy < 0) | (sy >= ny)
            if self.geometry == 2:
                solid = solid | (sz < 0) | (sz >= nz)
            sy, sz = sy % ny, sz % nz
            if self.geometry == 2:
                solid = solid | ~self.fluid_zy[sz[:, 0], sy[0].T.reshape(1, -1)][:, :, None]
            self.src[i] = torch.where(solid, opp[i] * N + here, i * N + sx + nx * (sy + ny * sz)).reshape(-1)
            if self.geometry == 1 and cx and cy:
                # f_opp meets the wall and comes back as f_i: minus 2 w rho (c_opp . u_w) / c_s^2
                row = 0 if cy > 0 else ny - 1
                self.wall.append((i, row, 6.0 / 36.0 * cx * lat.get('wall_u', [0, 0])[0 if cy > 0 else 1]))
        self.rho = torch.ones(N, dtype=F64, device=dev)
        self.u = torch.zeros(3, N, dtype=F64, device=dev) if u0 is None else torch.from_numpy(u0).to(dev)
        self.u = self.u * self.fluid
        self.f = self._equilibrium(self.rho, self.u)

    def _equilibrium(self, rho, u):
        cu = self.c @ u
        return self.wt[:, None] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def collide_stream(self, g):
        G = self.g0 + g if g is not None else self.g0.expand(3, self.rho.numel())
        f = self.f
        rho = f.sum(0)
        u = (self.c.T @ f + 0.5 * G) / rho
        rho, u = torch.where(self.fluid, rho, 1.0), torch.where(self.fluid, u, 0.0)
        cu, cG = self.c @ u, self.c @ G
        post = self.wt[:, None] * (3 * (cG - (u * G).sum(0)) + 9 * cu * cG) * (1 - 0.5 / self.tau)
        post += f + (self._equilibrium(rho, u) - f) / self.tau
        self.f = post.view(-1)[self.src]
        nx, ny, nz = self.n
        r = rho.view(nz, ny, nx)
        for i, row, k in self.wall:
            self.f[i].view(nz, ny, nx)[:, row] += k * r[:, row]
        self.rho, self.u = rho, u

    def fields(self):
        return self.rho * self.fluid, self.u * self.fluid


class _Membranes:
    """F = -dU/dX of red-cell membranes on one template, by automatic differentiation of the energy."""

    def __init__(self, mesh, bodies):
        dev = _device()
        tris = np.asarray(mesh['tris'], dtype=np.int64)
        wing = {}
        for t in tris:
            for s in range(3):
                wing[(int(t[s]), int(t[(s + 1) % 3]))] = int(t[(s + 2) % 3])
        E = np.array([(a, b, c, wing[(b, a)]) for (a, b), c in wing.items() if a < b])
        self.t, self.e = torch.from_numpy(tris).to(dev), torch.from_numpy(E).to(dev)
        self.p = {k: torch.tensor([b[k] for b in bodies], dtype=F64, device=dev)[:, None]
                  for k in ('kBT_p', 'k_b', 'k_l', 'k_g', 'k_v')}
        rest = torch.from_numpy(np.ascontiguousarray(mesh['rest_X'].T)).to(dev)[None]
        self.l0, self.th0, self.A0, self.V0 = (v[0] for v in self._shape(rest))

    def _shape(self, X):        # [B][V][3]
        a, b, c, d = (X[:, self.e[:, k]] for k in range(4))
        ev = b - a
        l = ev.norm(dim=2)
        n1, n2 = torch.linalg.cross(ev, c - a), torch.linalg.cross(a - b, d - b)
        th = torch.atan2((torch.linalg.cross(n1, n2) * ev).sum(2) / l, (n1 * n2).sum(2))
        p, q, r = (X[:, self.t[:, k]] for k in range(3))
        N = torch.linalg.cross(q - p, r - p)
        return l, th, 0.5 * N.norm(dim=2), (p * torch.linalg.cross(q, r)).sum((1, 2)) / 6

    def forces(self, X):        # [3][B V]
        B = self.p['k_b'].shape[0]
        out = []
        Xb = X.reshape(3, B, -1).permute(1, 2, 0)
        for s in range(0, B, 512):
            k = {n: v[s:s + 512] for n, v in self.p.items()}
            Y = Xb[s:s + 512]
            o = Y.mean(1, keepdim=True)
            Y = (Y - o).detach().requires_grad_(True)
            with torch.enable_grad():
                l, th, A, V = self._shape(Y)
                x = l / (2 * self.l0)
                U = (k['kBT_p'] * 0.5 * self.l0 * (3 * x ** 2 - 2 * x ** 3) / (1 - x)
                     + 1.25 * k['kBT_p'] * self.l0 ** 2 / l).sum()
                U = U + (k['k_b'] * (1 - torch.cos(th - self.th0))).sum()
                A0 = self.A0.sum()
                U = U + (k['k_l'] * (A - self.A0) ** 2 / (2 * self.A0)).sum()
                U = U + (k['k_g'][:, 0] * (A.sum(1) - A0) ** 2 / (2 * A0) + k['k_v'][:, 0] * (V - self.V0) ** 2 / (2 * self.V0)).sum()
                out.append(-torch.autograd.grad(U, Y)[0])
        return torch.cat(out).permute(2, 0, 1).reshape(3, -1)


def _filament_forces(X, bodies):      # [3][n b], all chains alike but for k_b
    n = len(bodies)
    dev = X.device
    kb = torch.tensor([b['k_b'] for b in bodies], dtype=F64, device=dev)[:, None]
    kt, l0 = bodies[0]['kBT_p'], bodies[0]['l0']
    Y = X.reshape(3, n, -1).permute(1, 2, 0).detach().requires_grad_(True)
    with torch.enable_grad():
        e = Y[:, 1:] - Y[:, :-1]
        l = e.norm(dim=2)
        x = l / (2 * l0)
        U = (kt * 0.5 * l0 * (3 * x ** 2 - 2 * x ** 3) / (1 - x) + 1.25 * kt * l0 ** 2 / l).sum()
        w = torch.linalg.cross(e[:, :-1], e[:, 1:])
        phi = torch.atan2(((w * w).sum(2) + 1e-300).sqrt(), (e[:, :-1] * e[:, 1:]).sum(2))
        U = U + (kb * phi ** 2).sum()
        F = -torch.autograd.grad(U, Y)[0]
    return F.permute(2, 0, 1).reshape(3, -1)


class _Morse:
    """Pairs of markers of different bodies within the cutoff, from a list with a margin."""

    def __init__(self, lat, bodies, k):
        dev = _device()
        self.k = k
        self.L = torch.tensor([lat['nx'], lat['ny'], lat['nz']], dtype=F64, device=dev)[:, None]
        self.periodic = torch.tensor([True, lat['geometry'] == 0, lat['geometry'] != 2], device=dev)[:, None]
        self.own = torch.cat([torch.full((b['count'],), i) for i, b in enumerate(bodies)]).to(dev)
        self.at = None

    def _apart(self, X, i, j):
        d = X[:, i] - X[:, j]
        return torch.where(self.periodic, d - self.L * torch.round(d / self.L), d)

    def _build(self, X):
        dev, reach = X.device, self.k['rc'] + 0.5
        nb = torch.clamp((self.L / reach).floor(), min=1)
        W = torch.where(self.periodic, X % self.L, X)
        b = torch.minimum(torch.clamp((W / self.L * nb).floor(), min=0), nb - 1).long()
        n = [int(v) for v in nb[:, 0]]
        key = b[0] + n[0] * (b[1] + n[1] * b[2])
        order = torch.argsort(key)
        start = torch.searchsorted(key[order], torch.arange(n[0] * n[1] * n[2] + 1, device=dev))
        pairs = []
        seen = torch.arange(X.shape[1], device=dev)
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    q = b + torch.tensor([[dx], [dy], [dz]], device=dev)
                    ok = (self.periodic | ((q >= 0) & (q < nb))).all(0)
                    q = q % nb.long()
                    kk = q[0] + n[0] * (q[1] + n[1] * q[2])
                    lo, cnt = start[kk], (start[kk + 1] - start[kk]) * ok
                    i = torch.repeat_interleave(seen, cnt)
                    first = torch.cumsum(cnt, 0) - cnt
                    j = order[lo[i] + torch.arange(i.numel(), device=dev) - first[i]]
                    keep = self.own[i] != self.own[j]
                    i, j = i[keep], j[keep]
                    near = (self._apart(X, i, j) ** 2).sum(0) < reach ** 2
                    pairs.append(torch.stack([i[near], j[near]]))
        self.pairs = torch.unique(torch.cat(pairs, 1), dim=1) if min(n) < 3 else torch.cat(pairs, 1)
        self.at = X.clone()

    def forces(self, X):
        if self.at is None or float(((X - self.at) ** 2).sum(0).max()) > 0.24 ** 2:
            self._build(X)
        i, j = self.pairs
        d = self._apart(X, i, j)
        r = (d * d).sum(0).sqrt()
        e = torch.exp(-self.k['alpha'] * (r - self.k['r0']))
        c = torch.where((r < self.k['rc']) & (r > 0), 2 * self.k['alpha'] * self.k['D0'] * (e * e - e) / r, 0.0)
        return torch.zeros_like(X).index_add_(1, i, c * d)


class _Rigid:
    def __init__(self, b, X):
        self.b, dev = b, X.device
        t = lambda k: torch.tensor(b[k], dtype=F64, device=dev)  # noqa: E731
        self.C, self.q, self.V, self.w, self.I = t('center'), t('quat'), t('vel'), t('omega'), t('inertia')
        self.r = self._R().T @ (X - self.C[:, None])

    def _R(self):
        w, x, y, z = self.q
        return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]).view(3, 3)

    def step(self, X, U):
        """Forces on the fluid and the markers' new positions; moves the body."""
        R = self._R()
        arm = R @ self.r
        direct = self.b['kind'] == 3
        if direct:
            f = self.b['kappa'] * (U - self.V[:, None] - torch.linalg.cross(self.w[:, None].expand_as(arm), arm, dim=0))
        else:
            f = self.b['kappa'] * (X - self.C[:, None] - arm)
        T = torch.linalg.cross(arm, f, dim=0).sum(1)
        self.V = self.V + f.sum(1) / self.b['mass']
        self.C = self.C + self.V
        wb = R.T @ self.w
        wb = wb + (R.T @ T - torch.linalg.cross(wb, self.I * wb)) / self.I
        self.w = R @ wb
        q0, qv = self.q[0], self.q[1:]
        dq = 0.5 * torch.cat([-(self.w * qv).sum()[None], q0 * self.w + torch.linalg.cross(self.w, qv)])
        self.q = self.q + dq
        self.q = self.q / self.q.norm()
        return -f, (self._R() @ self.r + self.C[:, None]) if direct else X


class _Coupled:
    def __init__(self, w):
        self.fluid = _Fluid(w['lattice'], w.get('u0'))
        self.X = torch.from_numpy(np.ascontiguousarray(w['X'])).to(_device())
        self.U, self.F = torch.zeros_like(self.X), torch.zeros_like(self.X)
        cells = [b for b in w['bodies'] if b['kind'] == 0]
        self.chains = [b for b in w['bodies'] if b['kind'] == 2]
        self.cells = _Membranes(w['mesh'], cells) if cells else None
        self.n_cell = sum(b['count'] for b in cells)
        rigid = [b for b in w['bodies'] if b['kind'] in (1, 3)]
        self.rigid = _Rigid(rigid[0], self.X) if rigid else None
        self.morse = _Morse(w['lattice'], w['bodies'], w['morse']) if w.get('morse') else None

    def forces(self):
        if self.rigid is not None:
            self.F, self.X = self.rigid.step(self.X, self.U)
        elif self.cells is not None:
            self.F = self.cells.forces(self.X[:, :self.n_cell])
            if self.chains:
                self.F = torch.cat([self.F, _filament_forces(self.X[:, self.n_cell:], self.chains)], 1)
        if self.morse is not None:
            self.F = self.F + self.morse.forces(self.X)

    def step(self):
        self.forces()
        s = _Nodes(self.fluid, self.X)
        g = None
        if self.rigid is not None or self.cells is not None:
            g = torch.zeros_like(self.fluid.u)
            for a in range(3):
                g[a].index_add_(0, s.i.view(-1), (s.w * self.F[a][:, None]).view(-1))
        self.fluid.collide_stream(g)
        self.U = torch.stack([(self.fluid.u[a][s.i] * s.w).sum(1) for a in range(3)])
        if not (self.rigid is not None and self.rigid.b['kind'] == 3):
            self.X = self.X + self.U

    def run(self, steps):
        for _ in range(steps):
            self.step()
        out = dict(X=self.X, U=self.U, F=self.F)
        out['rho'], out['u'] = self.fluid.fields()
        return out


def exact(case, seed):
    k = case['kind']
    with torch.no_grad():
        if k == 'spread':
            X, F, R = _spread(case, seed)
            G = _Grid(dict(case, tube_radius=R))
            X, F = torch.from_numpy(X).to(_device()), torch.from_numpy(F).to(_device())
            s = _Nodes(G, X)
            g = torch.zeros(3, case['nx'] * case['ny'] * case['nz'], dtype=F64, device=X.device)
            for a in range(3):
                g[a].index_add_(0, s.i.view(-1), (s.w * F[a][:, None]).view(-1))
            return g
        if k == 'stretch':
            w, fe = _stretch(case, seed)
            cells = _Membranes(w['mesh'], w['bodies'])
            X, fe = torch.from_numpy(w['X']).to(_device()), torch.from_numpy(fe).to(_device())
            v = torch.zeros_like(X)
            F = cells.forces(X)
            for _ in range(case['steps']):      # damped velocity Verlet, dt = 1, gamma = 0.05, mass 1
                v = v + 0.5 * (F + fe - 0.05 * v)
                X = X + v
                F = cells.forces(X)
                v = (v + 0.5 * (F + fe)) / (1 + 0.5 * 0.05)
            return dict(X=X, F=F)
        if k == 'serve':
            done = []
            for w in _served(case, seed):
                C = _Coupled(w)
                r = C.run(case['steps'])
                b = C.rigid
                pad = lambda v: torch.cat([v, torch.zeros(4 - len(v), dtype=F64, device=v.device)])  # noqa: E731
                r['pose'] = torch.stack([pad(b.C), b.q, pad(b.V), pad(b.w)])
                done.append(r)
            out = {n: torch.cat([r[n].reshape(-1) for r in done]) for n in ('rho', 'u', 'X', 'U')}
            out['pose'] = torch.cat([r['pose'] for r in done])
            return out
        if case['nx'] * case['ny'] * case.get('nz', case['ny']) > 3e7:
            return None
        C = _Coupled(dict(tube=_tube, channel=_channel, shear=_shear, tracers=_tracers)[k](case, seed))
        out = C.run(case['steps'])
        if k == 'tracers':
            del out['F']
        if k == 'shear':
            out['pose'] = torch.cat([C.rigid.C, C.rigid.q, C.rigid.V, C.rigid.w])
        if k == 'channel':
            del out['rho'], out['u']
        return out
