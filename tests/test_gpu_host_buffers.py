"""The arrays a caller hands to the C ABI may be any memory that a CUDA copy
takes: ordinary, pinned or device memory, below and above the sizes from which
the library touches the pages of ordinary memory before the copy (64 KiB, 16
MiB). The same values in each."""
import ctypes as C

import numpy as np
import pytest

from tests._cases import markers_inside

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('memory', ['pinned', 'device'])
@pytest.mark.parametrize('n', [12, 40, 132])  # rho 14 KB, 0.5 MB, 18.4 MB
def test_arrays_outside_ordinary_memory(cuda_lib, n, memory):
    import torch
    lat = dict(nx=n, ny=n, nz=n, tau=0.8, geometry=0, body_force=[1e-5, 0, 0])
    X = markers_inside(lat, n * n, 2)
    N, M = n ** 3, X.shape[1]
    lib, sim = cuda_lib.load(), cuda_lib.Simulation(lat)
    sim.set_markers(None, [], X)
    sim.step(3)
    rho, u = sim.fields()
    Xh, Uh, _ = sim.markers()

    def make(count):
        t = torch.zeros(count, dtype=torch.float64)
        return t.cuda() if memory == 'device' else t.pin_memory()

    def ptr(t):
        return C.c_void_p(t.data_ptr())

    r, v, x, U = make(N), make(3 * N), make(3 * M), make(3 * M)
    torch.cuda.synchronize()
    assert lib.ibm_lbm_get_fields(sim.h, ptr(r), ptr(v)) == cuda_lib.OK
    assert lib.ibm_lbm_get_markers(sim.h, ptr(x), ptr(U), None) == cuda_lib.OK
    for t, a in ((r, rho), (v, u), (x, Xh), (U, Uh)):
        assert np.array_equal(t.cpu().numpy(), np.ravel(a))
    assert lib.ibm_lbm_set_lattice(sim.h, ptr(r), ptr(v)) == cuda_lib.OK
    f = make(19 * N)
    torch.cuda.synchronize()
    assert lib.ibm_lbm_get_populations(sim.h, ptr(f)) == cuda_lib.OK
    assert np.array_equal(f.cpu().numpy(), np.ravel(sim.populations()))
