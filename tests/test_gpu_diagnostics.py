"""Sums of the last collision's moments: float sums on the device against
extended-precision sums of the same FP32 values."""
import numpy as np
import pytest

from paper_1704_04551_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('shape,geometry', [
    ((5, 4, 4), 0), ((33, 17, 21), 1), ((128, 4, 4), 0), ((128, 8, 4), 0), ((40, 31, 29), 2),
    ((211, 163, 149), 0),  # past 16 cells a thread, the grid's last turn partly filled
])
def test_sums_of_moments(cuda_lib, shape, geometry):
    """Up to 16 cells are summed in three floats each. Even two floats would keep
    a cell's share to 32 * 32 * 2^-48 of the largest term (the second's rounding,
    2^-24 of errors that are each 2^-24 of a partial sum of 32 terms): 4e-12 of
    the sum of magnitudes; the FP64 sums add far less."""
    nx, ny, nz = shape
    lat = dict(nx=nx, ny=ny, nz=nz, tau=0.8, geometry=geometry, body_force=[1e-6, 0.0, 0.0])
    if geometry == 1:
        lat['wall_u'] = [-0.01, 0.02]
    if geometry == 2:
        lat['tube_radius'] = 13.0
    rho, u = I.random_fields(shape, seed=5)
    sim = cuda_lib.Simulation(lat)
    sim.set_lattice(rho, u)
    sim.step(2)
    rho, u = sim.fields()
    fluid = np.asarray(rho).ravel() != 0.0
    w = (np.asarray(rho).ravel()[fluid] - 1.0).astype(np.longdouble)
    v = np.asarray(u).reshape(3, -1)[:, fluid].astype(np.longdouble)
    d = sim.diagnostics()
    n = int(fluid.sum())
    assert d['fluid_cells'] == n
    # the mass is n + sum(rho - 1), rounded once more
    assert abs(d['mass'] - (n + w.sum())) <= 4e-12 * np.abs(w).sum() + 2.0 ** -52 * n
    for a in range(3):
        p = (1 + w) * v[a]
        err, size = abs(d['momentum'][a] - p.sum()), np.abs(p).sum()
        assert err <= 4e-12 * size + 1e-300, (a, float(err / size))
    assert abs(d['umax'] - float(np.sqrt((v ** 2).sum(0).max()))) <= 1e-6 * d['umax']
