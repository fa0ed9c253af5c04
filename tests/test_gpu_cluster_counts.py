"""Couplings by clusters of thread blocks where the count of bodies changes
how they run (Sec. 2.3): one or two blocks on an SM, and the counts around
those the device holds at once (15 and 36 clusters on 152 SMs). The same steps
as the stage interface, which takes the separate kernels; tolerances as in
test_gpu_cluster.py."""
import numpy as np
import pytest

from paper_1704_04551_gb300 import inputs as I
from tests import test_gpu_solid
from tests._cases import rel_l2

pytestmark = pytest.mark.gpu

LAT = dict(nx=50, ny=48, nz=46, tau=0.8, geometry=0, body_force=[2e-6, -1e-6, 5e-7])


def _places(n):
    k = int(np.ceil(n ** (1 / 3)))
    i = np.arange(n)
    return (np.stack([i % k, i // k % k, i // (k * k)], 1) + 0.5) * [50 / k, 48 / k, 46 / k]


def _rigid(n, freq, direct):
    rng = np.random.default_rng(2)
    X, bodies, first = [], [], 0
    for c in _places(n):
        x, b = I.rigid_ellipsoid(c, (4.0, 3.5, 3.0), I.random_quaternion(rng), first, freq=freq, kappa=0.01,
                                 direct=direct)
        X.append(x)
        bodies.append(dict(b, vel=(1e-3 * rng.standard_normal(3)).tolist()))
        first += x.shape[1]
    return dict(lattice=LAT, mesh=None, bodies=bodies, X=np.concatenate(X, axis=1))


def _membranes(n, freq):
    rest, tris = I.rbc_rest_shape(9.0, freq)
    V = rest.shape[1]
    rng = np.random.default_rng(3)
    X = [rest * np.exp(rng.uniform(-0.05, 0.05, (3, 1))) + c[:, None] for c in _places(n)]
    bodies = [I._body(I.BODY_MEMBRANE, k * V, V, kBT_p=1e-3, k_b=5e-4, k_l=3e-3, k_g=2e-3, k_v=2e-3) for k in range(n)]
    return dict(lattice=LAT, mesh=dict(rest_X=rest, tris=tris), bodies=bodies, X=np.concatenate(X, axis=1))


def _match_stages(cuda_lib, w):
    a, b = cuda_lib.Simulation.from_workload(w), cuda_lib.Simulation.from_workload(w)
    for n in (1, 18):
        a.step(n)
        for _ in range(n):
            for st in (cuda_lib.STAGE_FORCES, cuda_lib.STAGE_SPREAD, cuda_lib.STAGE_COLLIDE, cuda_lib.STAGE_INTERP):
                b.stage(st)
    (Xa, _, Fa), (Xb, _, Fb) = a.markers(), b.markers()
    assert np.abs(Fa).max() > 1e-6
    assert rel_l2(a.fields()[1], b.fields()[1]) < 1e-6
    assert np.abs(Xa - Xb).max() < 1e-7
    assert np.abs(Fa - Fb).max() < 1e-4 * np.abs(Fb).max()
    assert np.abs(a.force_density()).max() == 0.0


@pytest.mark.parametrize('n,freq,direct', [(15, 4, False), (16, 4, False), (36, 4, True), (37, 4, True),
                                           (37, 6, False), (54, 6, False), (72, 8, False), (73, 8, False)])
def test_rigid_counts_match_stages(cuda_lib, n, freq, direct):
    _match_stages(cuda_lib, _rigid(n, freq, direct))


@pytest.mark.parametrize('n,freq', [(1, 4), (15, 6), (16, 6), (16, 8), (36, 8), (37, 8)])
def test_membrane_counts_match_stages(cuda_lib, n, freq):
    _match_stages(cuda_lib, _membranes(n, freq))


@pytest.mark.parametrize('n,freq,direct,clusters', [(30, 4, True, True), (200, 4, False, False), (200, 6, False, False),
                                                    (100, 6, True, False)])
def test_many_rigid_bodies_take_the_separate_kernels(cuda_lib, n, freq, direct, clusters):
    """Clusters need a second force density from the second step on; the
    separate kernels, which many bodies take, need none."""
    sim = cuda_lib.Simulation.from_workload(_rigid(n, freq, direct))
    held = sim.device_bytes
    sim.step(4)
    assert (sim.device_bytes - held >= 16 * sim.N) == clusters
    assert clusters or sim.device_bytes == held


# clusters in one wave, in two, and the general path
@pytest.mark.parametrize('freq,bodies', [(2, 15), (2, 30), (2, 31), (6, 45)])
def test_solid_counts_match_oracle(cuda_lib, freq, bodies):
    test_gpu_solid.test_solid_steps_of_several_bodies_match_oracle(cuda_lib, freq, bodies, (1, 7))


@pytest.mark.parametrize('rigids,clusters', [(20, True), (40, False)])
def test_rigid_bodies_beside_membranes(cuda_lib, rigids, clusters):
    r, m = _rigid(rigids, 6, False), _membranes(5, 4)
    n = r['X'].shape[1]
    X = np.concatenate([r['X'], m['X'] + 2.0], axis=1)
    w = dict(m, bodies=r['bodies'] + [dict(b, first=b['first'] + n) for b in m['bodies']], X=X)
    sim = cuda_lib.Simulation.from_workload(w)
    held = sim.device_bytes
    sim.step(4)
    assert (sim.device_bytes - held >= 16 * sim.N) == clusters
    _match_stages(cuda_lib, w)


@pytest.mark.parametrize('kind', ['rigid', 'cluster_membranes', 'fused_membranes'])
def test_no_memory_for_the_second_density(cuda_lib, kind):
    """An allocator that has nothing left when the first coupled step asks for
    the second force density: the same steps, one at a time."""
    import torch

    class Full(cuda_lib.TorchMemory):
        full = False

        def _on_alloc(self, nbytes, ctx):
            return None if self.full else super()._on_alloc(nbytes, ctx)

    w = _rigid(3, 4, False) if kind == 'rigid' else _membranes(3 if kind == 'cluster_membranes' else 40, 8)
    mem = Full(torch.device('cuda', 0))
    a, b = cuda_lib.Simulation.from_workload(w, memory=mem), cuda_lib.Simulation.from_workload(w)
    held = a.device_bytes
    mem.full = True
    for n in (2, 19):
        a.step(n)
        b.step(n)
    assert a.device_bytes == held
    mem.full = False
    (Xa, _, Fa), (Xb, _, Fb) = a.markers(), b.markers()
    assert np.abs(Xa - Xb).max() < 1e-7
    assert np.abs(Fa - Fb).max() < 1e-4 * np.abs(Fb).max()
    assert rel_l2(a.fields()[1], b.fields()[1]) < 1e-6
    assert np.abs(a.force_density()).max() == 0.0
