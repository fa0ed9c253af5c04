"""The half-precision collide with two cells per thread (Sec. 2.1, Eqs. lbm,
BGKequilibrium, rho_u, the Guo term), which lattices of 2^18 fluid cells and
more with even rows take: the shortest rows, rows that are no multiple of a
warp's cells, against the FP64 oracle: one even and one odd step from a random
state, three geometries, moving walls, a force density on some tiles. Each step rounds a stored population once (FP16: 2^-11 of its
scaled deviation, BF16: 2^-8), so two steps bound the error by about three
such roundings of the largest deviation (collision and streaming of the first
step's rounding included)."""
import numpy as np
import pytest

import oracle as O
from paper_1704_04551_gb300 import inputs as I
from tests._cases import fluid_mask, markers_inside, shape

pytestmark = pytest.mark.gpu
EPS = {'f16': 2.0 ** -11, 'bf16': 2.0 ** -8}


@pytest.mark.parametrize('storage', list(EPS))
@pytest.mark.parametrize('nx,ny,nz', [(4, 292, 290), (62, 75, 74), (130, 52, 51)])
@pytest.mark.parametrize('geometry', [0, 1, 2])
def test_even_rows_match_oracle(cuda_lib, geometry, nx, ny, nz, storage):
    lat = dict(nx=nx, ny=ny, nz=nz, tau=0.8, geometry=geometry, wall_u=[-0.015, 0.02], tube_radius=0.5 * ny - 0.6,
               body_force=[2e-5, -1e-5, 5e-6])
    sim, ora = cuda_lib.Simulation(lat, storage=storage), O.Oracle(lat)
    fl = fluid_mask(lat)
    assert fl.sum() >= 1 << 18
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    scale = np.array([4.0] + [16.0] * 6 + [32.0] * 12)
    rng = np.random.default_rng(geometry * 100 + nx)
    # deviations that the storage holds exactly
    dev = np.round(rng.uniform(-0.02, 0.02, (19, sim.N)) * 2 ** 11) / 2 ** 11 / 4.0
    if storage == 'bf16':
        dev = np.round(rng.uniform(-0.02, 0.02, (19, sim.N)) * 2 ** 10) / 2 ** 10 / 4.0
    f0 = w[:, None] + dev * (4.0 / scale)[:, None]
    f0[:, ~fl] = 0.0
    X = markers_inside(lat, 5, 3)
    F = 1e-4 * rng.standard_normal((3, 5))
    for s in (sim, ora):
        s.set_populations(f0)
    sim.set_markers(None, [], X)
    ora.set_bodies([], X)
    sim.set_marker_forces(F)
    ora.set_marker_forces(F)
    largest = np.abs(dev).max() * 4.0
    for step in range(2):
        sim.stage(cuda_lib.STAGE_SPREAD)
        ora.stage_spread()
        sim.stage(cuda_lib.STAGE_COLLIDE)
        ora.stage_collide_stream()
        fg, fo = sim.populations()[:, fl], ora.populations()[:, fl]
        # stored (scaled) deviations, in units of one rounding of the largest
        err = (np.abs(fg - fo) * scale[:, None]).max() / (EPS[storage] * max(largest, np.abs((fo - w[:, None]) * scale[:, None]).max()))
        assert err < 1.0 + 3.0 * step, (step, err)
        assert np.abs(sim.fields()[1][:, fl] - ora.fields()[1][:, fl]).max() < 20 * (1e-7 + step * EPS[storage] * largest)
        sim.stage(cuda_lib.STAGE_INTERP)
        ora.stage_interpolate()
