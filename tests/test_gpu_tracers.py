"""Passive tracers in ibm_lbm_step (Sec. 2.3, Eq. ibmVelocityInterpret): few
of them (their tiles are marked), many (the collision writes every velocity),
beside a rigid body and a membrane, ragged group sizes, against the oracle, and
with forces left by the stage interface, which a step zeroes. Tolerances as in
test_gpu_parity.py."""
import numpy as np
import pytest

import oracle as O
from paper_1704_04551_gb300 import inputs as I
from tests._cases import LATTICES, fluid_mask, markers_inside, membrane_case, rel_l2, shape

pytestmark = pytest.mark.gpu


def _check(sim, ora, lat, steps):
    sim.step(steps)
    ora.step(steps)
    fl = fluid_mask(lat)
    assert rel_l2(sim.fields()[1][:, fl], ora.fields()[1][:, fl]) < 1e-5
    Xg, Ug, Fg = sim.markers()
    Xo, Uo, _ = ora.markers()
    assert np.abs(Xg - Xo).max() < 1e-5
    assert rel_l2(Ug, Uo) < 1e-4
    return Fg


# tiles of these lattices: 18-32, so that 1-4 tracers are marked, 257 and more not
@pytest.mark.parametrize('M', [1, 4, 257, 1000])
@pytest.mark.parametrize('geom', list(LATTICES))
def test_tracers_match_oracle(cuda_lib, geom, M):
    lat = LATTICES[geom]
    X = markers_inside(lat, M, 3)
    rho, u = I.random_fields(shape(lat), 8, u_amp=0.01, rho_amp=0.002)
    sim, ora = cuda_lib.Simulation(lat), O.Oracle(lat)
    sim.set_lattice(rho, u)
    ora.set_equilibrium(rho, u)
    sim.set_markers(None, [], X)
    ora.set_bodies([], X)
    sim.set_marker_forces(1e-3 * np.ones((3, M)))  # a step zeroes the forces on tracers
    F = _check(sim, ora, lat, 21)
    assert np.abs(F).max() == 0.0


@pytest.mark.parametrize('M', [7, 3000])
def test_tracers_beside_bodies_match_oracle(cuda_lib, M):
    w = membrane_case()
    lat = dict(w['lattice'], body_force=[2e-6, 0, 0])
    n = w['X'].shape[1]
    R, rigid = I.rigid_ellipsoid([20.0, 30.0, 19.0], (3.0, 2.0, 2.0), [1.0, 0.0, 0.0, 0.0], n, freq=3)
    rng = np.random.default_rng(2)
    r, th = 14.0 * np.sqrt(rng.random(M)), 2 * np.pi * rng.random(M)
    T = np.stack([40 * rng.random(M), 19.5 + r * np.cos(th), 19.5 + r * np.sin(th)])
    w = dict(w, lattice=lat, bodies=w['bodies'] + [rigid], X=np.concatenate([w['X'], R, T], axis=1))
    F = _check(cuda_lib.Simulation.from_workload(w), O.Oracle.from_workload(w), lat, 20)
    assert np.abs(F[:, -M:]).max() == 0.0 and np.abs(F[:, :n]).max() > 0.0


@pytest.mark.parametrize('packed', [True, False])
def test_many_tracers_of_a_large_lattice_match_stages(cuda_lib, packed):
    """Past 2^23 cells packed tracers are marked, scattered ones are not; the
    stage interface, which computes every velocity, moves them the same way
    (the same arithmetic; populations FP32 in both)."""
    lat = dict(nx=256, ny=188, nz=178, tau=0.8, geometry=0, body_force=[2e-6, -1e-6, 5e-7])
    n = np.array(shape(lat), float)[:, None]
    M = 4400  # tiles: 16920
    rng = np.random.default_rng(5)
    X = (0.5 * n + 6.0 * (2 * rng.random((3, M)) - 1)) if packed else n * rng.random((3, M))
    X[:, :40] = rng.uniform(-3.0, 3.0, (3, 40))  # a few across the boundaries
    u = 0.02 * rng.standard_normal((3, 1)) * np.ones((3, int(n.prod())))
    a, b = cuda_lib.Simulation(lat), cuda_lib.Simulation(lat)
    for s in (a, b):
        s.set_lattice(None, u)
        s.set_markers(None, [], X)
    a.step(5)
    for _ in range(5):
        for st in (cuda_lib.STAGE_FORCES, cuda_lib.STAGE_SPREAD, cuda_lib.STAGE_COLLIDE, cuda_lib.STAGE_INTERP):
            b.stage(st)
    (Xa, Ua, _), (Xb, Ub, _) = a.markers(), b.markers()
    assert np.abs(Xa - X).max() > 1e-3
    assert np.abs(Xa - Xb).max() < 1e-7 and rel_l2(Ua, Ub) < 1e-6
    assert rel_l2(a.fields()[1], b.fields()[1]) < 1e-6
