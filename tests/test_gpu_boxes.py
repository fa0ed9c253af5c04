"""Stencil boxes larger than a thread block's shared memory, processed in
slabs of z layers (Sec. 2.3, Eqs. ibmForceSpread, ibmVelocityInterpret): in the
fused coupling kernel of membranes, and in both families of the separate
transfer kernels; whole boxes and boxes beyond the slabs' limit beside them.
Tolerances as in test_gpu_parity.py and test_gpu_parity_paths.py."""
import numpy as np
import pytest

import oracle as O
from paper_1704_04551_gb300 import inputs as I
from tests._cases import WIDE, cluster_tracers, rel_l2, shape

pytestmark = pytest.mark.gpu


def _cells(diameter, n, lat, seed):
    """n red cells of one template at random orientations and places."""
    rest, tris = I.rbc_rest_shape(diameter, 8)
    V = rest.shape[1]
    rng = np.random.default_rng(seed)
    X, bodies = [], []
    for k in range(n):
        c = rng.random(3) * np.array(shape(lat))
        R = I.quat_to_matrix(I.random_quaternion(rng))
        X.append(R @ (rest * np.exp(rng.uniform(-0.05, 0.05, (3, 1)))) + c[:, None])
        bodies.append(I._body(I.BODY_MEMBRANE, k * V, V, kBT_p=1e-4, k_b=5e-5, k_l=3e-3, k_g=2e-3, k_v=2e-3))
    return dict(lattice=lat, mesh=dict(rest_X=rest, tris=tris), bodies=bodies, X=np.concatenate(X, axis=1))


# one block per body (the count is above the clusters' range): boxes around
# the shared-memory limit, all in slabs, and some beyond the slabs
@pytest.mark.parametrize('diameter', [17.0, 24.0, 44.0])
def test_fused_membranes_with_large_boxes(cuda_lib, diameter):
    lat = dict(nx=96, ny=90, nz=94, tau=1.0, geometry=0, body_force=[2e-6, 0, 0])
    w = _cells(diameter, 50, lat, 5)
    a, b = cuda_lib.Simulation.from_workload(w), cuda_lib.Simulation.from_workload(w)
    a.step(19)
    for _ in range(19):
        for st in (cuda_lib.STAGE_FORCES, cuda_lib.STAGE_SPREAD, cuda_lib.STAGE_COLLIDE, cuda_lib.STAGE_INTERP):
            b.stage(st)
    ora = O.Oracle.from_workload(w)
    ora.step(19)
    for s in (a, b):
        X, _, F = s.markers()
        Xo, _, Fo = ora.markers()
        assert rel_l2(s.fields()[1], ora.fields()[1]) < 1e-5
        assert np.abs(X - Xo).max() < 1e-5
        assert np.abs(F - Fo).max() < 1e-3 * np.abs(Fo).max()
        assert np.abs(s.force_density()).max() == 0.0


@pytest.mark.parametrize('n_clusters', [40, 600])
@pytest.mark.parametrize('geom', list(WIDE))
def test_transfer_in_slabs(cuda_lib, geom, n_clusters):
    """Tracer groups packed into cubes of 18 lu (boxes of ~22^3 cells), few
    and many groups, against the oracle."""
    lat = dict(WIDE[geom])
    if geom == 'tube':
        lat.update(ny=60, nz=60, tube_radius=28.5)
    X, F = cluster_tracers(lat, n_clusters, 71 + n_clusters, half=9.0)
    sim, ora = cuda_lib.Simulation(lat), O.Oracle(lat)
    sim.set_markers(None, [], X)
    ora.set_bodies([], X)
    sim.set_marker_forces(F)
    ora.set_marker_forces(F)
    sim.stage(cuda_lib.STAGE_SPREAD)
    ora.stage_spread()
    gg, go = sim.force_density(), ora.force_density()
    assert np.abs(gg - go).max() < 2e-5 * np.abs(go).max()
    rho, u = I.random_fields(shape(lat), 32)
    sim.set_lattice(rho, u)
    ora.set_equilibrium(rho, u)
    sim.stage(cuda_lib.STAGE_INTERP)
    ora.stage_interpolate()
    Xg, Ug, _ = sim.markers()
    Xo, Uo, _ = ora.markers()
    assert np.abs(Ug - Uo).max() < 2e-5 * np.abs(Uo).max()
    assert np.abs(Xg - Xo).max() < 1e-6


# spheres around the size from which boxes are no longer worth slabs: with four
# lanes a marker by their markers (362 and 812), with one block a membrane far
# beyond (whose layers also leave the fewest new layers in a slab)
@pytest.mark.parametrize('kind,n,freq,R', [('rigid', 75, 6, 7.3), ('rigid', 75, 6, 8.6), ('rigid', 75, 9, 9.5),
                                           ('rigid', 75, 9, 10.6), ('membrane', 40, 3, 13.4), ('membrane', 40, 3, 14.2)])
def test_spheres_around_the_slab_limit(cuda_lib, kind, n, freq, R):
    S, tris = I.geodesic_sphere(freq)
    V = S.shape[0]
    rest = (R * S).T.copy()
    lat = dict(nx=96, ny=90, nz=94, tau=1.0, geometry=0, body_force=[2e-6, 0, 0])
    rng = np.random.default_rng(8)
    C = rng.random((n, 3)) * [96, 90, 94]
    if kind == 'membrane':
        X = [rest * np.exp(rng.uniform(-0.02, 0.02, (3, 1))) + c[:, None] for c in C]
        bodies = [I._body(I.BODY_MEMBRANE, k * V, V, kBT_p=1e-4, k_b=5e-5, k_l=3e-3, k_g=2e-3, k_v=2e-3)
                  for k in range(n)]
        mesh = dict(rest_X=rest, tris=tris)
    else:
        X, bodies, mesh = [], [], None
        for k, c in enumerate(C):
            x, b = I.rigid_ellipsoid(c, (R, R, R), I.random_quaternion(rng), k * V, freq=freq, kappa=0.02)
            X.append(x)
            bodies.append(dict(b, vel=(1e-3 * rng.standard_normal(3)).tolist()))
    w = dict(lattice=lat, mesh=mesh, bodies=bodies, X=np.concatenate(X, axis=1))
    sim, ora = cuda_lib.Simulation.from_workload(w), O.Oracle.from_workload(w)
    sim.step(5)
    ora.step(5)
    (Xg, _, Fg), (Xo, _, Fo) = sim.markers(), ora.markers()
    assert rel_l2(sim.fields()[1], ora.fields()[1]) < 1e-5
    assert np.abs(Xg - Xo).max() < 1e-5
    assert np.abs(Fg - Fo).max() < 1e-3 * np.abs(Fo).max()
    assert np.abs(sim.force_density()).max() == 0.0
