"""The coupling of few bodies by clusters of thread blocks (Sec. 2.3: Eqs.
ibmForceSpread, ibmVelocityInterpret; Sec. 2.2 for membranes): the same steps
as the stage interface, which spreads and interpolates with the separate
kernels. Sizes at the edges of the split: fewer markers than blocks, one more
than a multiple, the largest count a body may have, bodies across periodic
boundaries and against a wall, a body whose boxes do not fit shared memory
(global atomics), one whose parts are too far apart for a common box, one large
enough that all warps clear its box, several bodies that share cells, odd starts and single
steps.

Tolerances as in test_gpu_parity.py: both paths do the same arithmetic on
the same integers, and differ where bodies add into a shared cell in another
order (float atomics)."""
import numpy as np
import pytest

import oracle as O
from paper_1704_04551_gb300 import inputs as I
from tests._cases import rel_l2

pytestmark = pytest.mark.gpu


def _rigid(lat, bodies):
    """Rigid bodies from (count, centre, spread, direct): markers on a random ellipsoid."""
    rng = np.random.default_rng(7)
    X, out, first = [], [], 0
    for count, centre, size, direct in bodies:
        d = rng.standard_normal((3, count))
        x = np.array(centre, float)[:, None] + np.array(size, float)[:, None] * d / np.linalg.norm(d, axis=0)
        X.append(x)
        mass = 200.0
        inertia = [mass * f * max(size) ** 2 / 5 for f in (1.6, 1.8, 2.0)]
        out.append(I._body(I.BODY_RIGID_DIRECT if direct else I.BODY_RIGID, first, count,
                           kappa=(60.0 if direct else 8.0) / count, mass=mass, inertia=inertia,
                           center=list(map(float, centre)), vel=[1e-3, -5e-4, 2e-4], omega=[1e-3, 2e-3, -1e-3]))
        first += count
    return dict(lattice=lat, mesh=None, bodies=out, X=np.concatenate(X, axis=1))


PER = dict(nx=40, ny=28, nz=26, tau=0.8, geometry=0, body_force=[2e-6, -1e-6, 5e-7])
WALL = dict(nx=33, ny=27, nz=30, tau=0.7, geometry=1, wall_u=[-0.01, 0.015], body_force=[0, 0, 0])
TUBE = dict(nx=37, ny=30, nz=30, tau=1.0, geometry=2, tube_radius=13.5, body_force=[3e-6, 0, 0])
WIDE = dict(nx=96, ny=90, nz=88, tau=0.8, geometry=0, body_force=[1e-6, 0, 0])
CASES = {
    'fewer_markers_than_blocks': (PER, [(5, (20, 14, 13), (4, 4, 4), False)]),
    'one_over_a_multiple': (TUBE, [(57, (10, 14, 15), (4, 3, 3), False)]),
    'largest_body': (WALL, [(4096, (16, 13, 15), (7, 6, 6), False)]),
    'across_boundaries': (PER, [(300, (0.5, 27.5, 1.0), (5, 4, 3), False)]),
    'against_a_wall': (WALL, [(812, (16, 2.0, 15), (6, 3, 3), True)]),
    'direct_and_tether_sharing_cells': (TUBE, [(812, (12, 14, 15), (6, 4, 4), True), (400, (18, 15, 14), (4, 4, 4), False)]),
    'eighths_far_apart': (WIDE, [(8, (48, 45, 44), (70, 60, 60), False)]),
    'large_body': (WIDE, [(812, (40, 45, 44), (19, 9, 8), False)]),
    'boxes_too_large': (WIDE, [(640, (48, 45, 44), (40, 38, 37), False)]),
}


@pytest.mark.parametrize('name', list(CASES))
def test_rigid_clusters_match_stages(cuda_lib, name):
    lat, bodies = CASES[name]
    w = _rigid(lat, bodies)
    a, b = cuda_lib.Simulation.from_workload(w), cuda_lib.Simulation.from_workload(w)
    # single steps, an odd start, a call long enough for a captured chunk
    for n in (1, 2, 18, 1, 3):
        a.step(n)
        for _ in range(n):
            for st in (cuda_lib.STAGE_FORCES, cuda_lib.STAGE_SPREAD, cuda_lib.STAGE_COLLIDE, cuda_lib.STAGE_INTERP):
                b.stage(st)
    Xa, Ua, Fa = a.markers()
    Xb, Ub, Fb = b.markers()
    assert np.abs(Fa).max() > 1e-6
    assert rel_l2(a.fields()[1], b.fields()[1]) < 1e-6
    assert np.abs(Xa - Xb).max() < 1e-7
    assert np.abs(Fa - Fb).max() < 1e-4 * np.abs(Fb).max()
    for p, q in zip(a.bodies(), b.bodies()):
        for k in ('center', 'quat', 'vel', 'omega'):
            assert np.allclose(p[k], q[k], rtol=1e-5, atol=1e-9), k
    assert np.abs(a.force_density()).max() == 0.0  # consumed and cleared
    assert a.diagnostics()['steps'] == 25


@pytest.mark.parametrize('freq', [1, 2, 16])
def test_membrane_clusters_match_stages(cuda_lib, freq):
    """The smallest templates (12 and 42 vertices: two and six per block)
    against the stages, and a large one (2562 vertices) against the oracle:
    the separate kernels spread it in three groups, each with a fixed-point
    scale of its own, so their integers are others. Two bodies that share
    cells."""
    rest, tris = I.rbc_rest_shape(12.0, freq)
    V = rest.shape[1]
    rng = np.random.default_rng(3)
    X = np.concatenate([1.05 * rest + [[12.0], [14.0], [13.0]], 0.96 * rest + [[14.0], [13.0], [19.0]]], axis=1)
    X += 0.01 * rng.standard_normal(X.shape)
    bodies = [I._body(I.BODY_MEMBRANE, k * V, V, kBT_p=1e-3, k_b=5e-4, k_l=3e-3, k_g=2e-3, k_v=2e-3) for k in range(2)]
    w = dict(lattice=PER, mesh=dict(rest_X=rest, tris=tris), bodies=bodies, X=X)
    a, b = cuda_lib.Simulation.from_workload(w), cuda_lib.Simulation.from_workload(w)
    ora = O.Oracle.from_workload(w)
    for n in (1, 19):
        a.step(n)
        for _ in range(n):
            for st in (cuda_lib.STAGE_FORCES, cuda_lib.STAGE_SPREAD, cuda_lib.STAGE_COLLIDE, cuda_lib.STAGE_INTERP):
                b.stage(st)
    ora.step(20)
    Xo, _, Fo = ora.markers()
    Xa, _, Fa = a.markers()
    assert rel_l2(a.fields()[1], ora.fields()[1]) < 1e-5
    assert np.abs(Xa - Xo).max() < 1e-5
    assert np.abs(Fa - Fo).max() < 1e-3 * np.abs(Fo).max()
    if V > 1024:
        return
    Fb = b.markers()[2]
    assert np.abs(Fa).max() > 1e-6
    assert rel_l2(a.fields()[1], b.fields()[1]) < 1e-6
    assert np.abs(a.markers()[0] - b.markers()[0]).max() < 1e-7
    assert np.abs(Fa - Fb).max() < 1e-4 * np.abs(Fb).max()
