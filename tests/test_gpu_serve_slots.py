"""Servers of few and of many slots: clusters couple the bodies of few, the
separate kernels those of many (csrc/api.cu, rigid_clusters_max). The same
cases in both, against the single-lattice handle, within the bounds of
test_gpu_serve.py; within one server a case's result does not depend on what
else it serves (bit for bit where one marker group covers all markers). Clusters
hold a second force density, 16 bytes a cell, so the memory shows the path."""
import numpy as np
import pytest

from paper_1704_04551_gb300 import inputs as I
from tests._cases import rel_l2

pytestmark = pytest.mark.gpu


def _cell(seed):
    return I.shear_ellipsoid(n=32, axes=(5.0, 2.5, 2.5), seed=seed)


def _serve(cuda_lib, cases, slots):
    import torch
    mem = cuda_lib.TorchMemory(torch.device('cuda', 0))
    srv = cuda_lib.Server(1 << 34, max_active=slots, chunk_steps=8, memory=mem)
    ids = [srv.submit(w, n) for w, n in cases]
    held = 0
    while True:
        rc, running, pending, _ = srv.advance()
        assert rc == cuda_lib.OK
        held = max(held, sum(t.numel() for t in mem.live.values()))
        if running == 0 and pending == 0:
            break
    out = [srv.result(i) for i in ids]
    srv.close()
    return out, held


@pytest.mark.parametrize('few,many', [(64, 65)])
def test_slots_choose_the_path(cuda_lib, few, many):
    # the first case runs longer than the others: alone in the last chunks
    cases = [(_cell(41), 70)] + [(_cell(50 + k), 33 + k) for k in range(3)]
    a, held_few = _serve(cuda_lib, cases, few)
    b, held_many = _serve(cuda_lib, cases, many)
    alone, _ = _serve(cuda_lib, cases[:1], many)
    N = 32 ** 3
    assert held_few - held_many >= 3 * 16 * N  # (four cases; boxes beside them)
    for k in ('rho', 'u', 'X', 'U'):
        assert np.array_equal(b[0][k], alone[0][k]), k
    for (w, n), p, q in zip(cases, a, b):
        sim = cuda_lib.Simulation.from_workload(w)
        sim.step(n)
        u, X = sim.fields()[1], sim.markers()[0]
        for r in (p, q):
            assert rel_l2(r['u'], u) < 1e-6
            assert np.abs(r['X'] - X).max() < 1e-7
