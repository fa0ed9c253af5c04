"""Membrane forces (Sec. 2.2, Eqs. inPlanePotential, areaConstraint,
volumeConstraint) where fixed point runs out of range: contributions so small
that no finite scale makes integers of them, and bodies whose area or volume is
thousands of times that at rest. One block per body and clusters, against the
oracle. The forces are FP32 sums of up to some tens of contributions: a
component's error is below 1e-3 of the largest one (test_gpu_parity.py)."""
import numpy as np
import pytest

import oracle as O
from paper_1704_04551_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LAT = dict(nx=32, ny=32, nz=32, tau=1.0, geometry=0, body_force=[0.0, 0.0, 0.0])


def _bodies(n, swell, factor):
    """n deformed red cells (162 vertices), `swell` times their rest size, moduli times `factor`."""
    rest, tris = I.rbc_rest_shape(10.0, 4)
    V = rest.shape[1]
    rng = np.random.default_rng(9)
    X = [swell * (rest * np.exp(rng.uniform(-0.05, 0.05, (3, 1)))) + 16.0 + 0.02 * rng.standard_normal(rest.shape)
         for _ in range(n)]
    moduli = dict(kBT_p=2e-3, k_b=1e-3, k_l=5e-3, k_g=4e-3, k_v=3e-3)
    bodies = [I._body(I.BODY_MEMBRANE, b * V, V, **{k: v * factor for k, v in moduli.items()}) for b in range(n)]
    return dict(lattice=LAT, mesh=dict(rest_X=rest, tris=tris), bodies=bodies, X=np.concatenate(X, axis=1))


def _forces_match(cuda_lib, w):
    sim, ora = cuda_lib.Simulation.from_workload(w), O.Oracle.from_workload(w)
    ora.stage_forces()
    Fo = ora.markers()[2]
    for _ in range(2):  # without and with a largest contribution of the evaluation before
        sim.stage(cuda_lib.STAGE_FORCES)
        F = sim.markers()[2]
        assert np.abs(F - Fo).max() < 1e-3 * np.abs(Fo).max()


# 2 bodies take clusters, 40 a block each
@pytest.mark.parametrize('n', [2, 40])
@pytest.mark.parametrize('factor', [1e-32, 1e-28, 1e-22])
def test_tiny_forces(cuda_lib, n, factor):
    _forces_match(cuda_lib, _bodies(n, 1.0, factor))


@pytest.mark.parametrize('n', [2, 40])
@pytest.mark.parametrize('swell', [20.0, 70.0, 300.0])
def test_swollen_cells(cuda_lib, n, swell):
    _forces_match(cuda_lib, _bodies(n, swell, 1.0))
