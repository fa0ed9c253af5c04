"""A force density that a SPREAD stage left is applied by the next
ibm_lbm_step, once, and is gone after it (Sec. 2.3, Eq. ibmForceSpread): the
way to push the fluid at markers outside bodies. Few tracers and many, rigid
bodies and membranes on every step path, both AA parities, the per-stage
timing, against the oracle, whose first step spreads the bodies' own forces and
these together. Tolerances as in test_gpu_parity.py."""
import numpy as np
import pytest

import oracle as O
from paper_1704_04551_gb300 import inputs as I
from tests._cases import LATTICES, fluid_mask, markers_inside, rel_l2

pytestmark = pytest.mark.gpu


def _oracle_step(ora, F_ext):
    ora.stage_forces()
    F = ora.markers()[2] + F_ext
    ora.set_marker_forces(F)
    ora.stage_spread()
    ora.stage_collide_stream()
    ora.stage_interpolate()


def _check(sim, ora, lat):
    fl = fluid_mask(lat)
    assert rel_l2(sim.fields()[1][:, fl], ora.fields()[1][:, fl]) < 1e-5
    (Xg, Ug, _), (Xo, Uo, _) = sim.markers(), ora.markers()
    assert np.abs(Xg - Xo).max() < 1e-5
    assert rel_l2(Ug, Uo) < 1e-4
    assert np.abs(sim.force_density()).max() == 0.0


def _run(cuda_lib, w, before, after, timed=False):
    """`before` steps, a SPREAD of forces, `after` steps (each a call)."""
    sim, ora = cuda_lib.Simulation.from_workload(w), O.Oracle.from_workload(w)
    if timed:
        sim.set_timing(64)
    if before:
        sim.step(before)
        ora.step(before)
    # forces that differ from marker to marker, a few per cent of what drives |u| to 0.1
    F = 2e-3 * np.random.default_rng(4).standard_normal(w['X'].shape)
    sim.set_marker_forces(F)
    sim.stage(cuda_lib.STAGE_SPREAD)
    assert np.abs(sim.force_density()).max() > 1e-5
    for n in after:
        sim.step(n)
        if F is not None:
            _oracle_step(ora, F)
            F, n = None, n - 1
        if n:
            ora.step(n)
        _check(sim, ora, w['lattice'])


# tiles of these lattices: 18-32, so that 4 tracers are marked, 1000 not
@pytest.mark.parametrize('before,after', [(0, (1, 3)), (1, (20,))])
@pytest.mark.parametrize('M', [4, 1000])
@pytest.mark.parametrize('geom', list(LATTICES))
def test_spread_then_step_with_tracers(cuda_lib, geom, M, before, after):
    lat = LATTICES[geom]
    _run(cuda_lib, dict(lattice=lat, bodies=[], X=markers_inside(lat, M, 3)), before, after)


@pytest.mark.parametrize('M', [4, 1000])
def test_spread_then_timed_step_with_tracers(cuda_lib, M):
    lat = LATTICES['ywalls']
    _run(cuda_lib, dict(lattice=lat, bodies=[], X=markers_inside(lat, M, 3)), 0, (1, 3), timed=True)


def test_spread_collide_then_step_leaves_no_density(cuda_lib):
    lat = LATTICES['periodic']
    sim = cuda_lib.Simulation(lat)
    sim.set_markers(None, [], markers_inside(lat, 9, 3))
    sim.set_marker_forces(1e-3 * np.ones((3, 9)))
    sim.stage(cuda_lib.STAGE_SPREAD)
    sim.stage(cuda_lib.STAGE_COLLIDE)
    sim.step(2)
    assert np.abs(sim.force_density()).max() == 0.0


def _tethered():
    lat = LATTICES['tube']
    X, body = I.rigid_ellipsoid([18.0, 6.5, 6.0], (3.0, 2.0, 2.0), [1.0, 0.0, 0.0, 0.0], 0, freq=3, kappa=0.05)
    return dict(lattice=lat, mesh=None, bodies=[dict(body, vel=[1e-3, 5e-4, 0.0])], X=X)


def _membranes(n):
    """n red cells of a coarse template (42 vertices): clusters, or from 39 on the fused kernel."""
    lat = dict(nx=40, ny=28, nz=26, tau=0.8, geometry=0, body_force=[2e-6, -1e-6, 5e-7])
    rest, tris = I.rbc_rest_shape(8.0, 2)
    V = rest.shape[1]
    rng = np.random.default_rng(6)
    C = rng.random((n, 3)) * [40, 28, 26]
    X = np.concatenate([1.04 * rest + c[:, None] + 0.01 * rng.standard_normal(rest.shape) for c in C], axis=1)
    bodies = [I._body(I.BODY_MEMBRANE, k * V, V, kBT_p=1e-3, k_b=5e-4, k_l=3e-3, k_g=2e-3, k_v=2e-3)
              for k in range(n)]
    return dict(lattice=lat, mesh=dict(rest_X=rest, tris=tris), bodies=bodies, X=X)


BODIES = dict(rigid=_tethered, cluster_membranes=lambda: _membranes(3), fused_membranes=lambda: _membranes(40))


@pytest.mark.parametrize('before,after', [(0, (2, 20)), (1, (1, 2)), (1, (20,)), (3, (3,))])
@pytest.mark.parametrize('kind', list(BODIES))
def test_spread_then_step_with_bodies(cuda_lib, kind, before, after):
    """Both parities: a coupled step's buffer goes with the parity, the stage's does not."""
    _run(cuda_lib, BODIES[kind](), before, after)


@pytest.mark.parametrize('M', [7, 45000])
def test_spread_then_step_with_tracers_beside_a_body(cuda_lib, M):
    """Tracers in the bodies' kernels (few) and in kernels of their own (more
    blocks than the device's SMs take beside the body's)."""
    w = _tethered()
    T = markers_inside(w['lattice'], M, 3)
    w = dict(w, X=np.concatenate([w['X'], T], axis=1))
    # (the same force on a cell for any number of tracers)
    F = 2e-3 / max(1.0, M / 1000.0) * np.random.default_rng(4).standard_normal(w['X'].shape)
    sim, ora = cuda_lib.Simulation.from_workload(w), O.Oracle.from_workload(w)
    for before, n in ((1, 3), (2, 18)):
        sim.step(before)
        ora.step(before)
        sim.set_marker_forces(F)
        sim.stage(cuda_lib.STAGE_SPREAD)
        sim.step(n)
        _oracle_step(ora, F)
        ora.step(n - 1)
        _check(sim, ora, w['lattice'])
