"""The accuracy of the sums of moments: terms that cancel to a remainder which
three floats hold and two lose. Moments as set_lattice stores them (FP32), one
thread block, so that a thread adds the eight cells of its column."""
import math

import numpy as np
import pytest

THREADS, CELLS = 256, 8  # cells t, t + 256, ... of a thread


def _column(rng):
    """a, b, c, t, -a, -b, -c, 0 for each thread: a in [1/2, 1), b and c of
    2^-12 and 2^-9 of that size with bits far below a's last one, t some units
    of 2^-52: the remainder."""
    f = np.float32
    a = (rng.integers(2 ** 23, 2 ** 24, THREADS) * 2.0 ** -24).astype(f)
    b = (rng.integers(2 ** 23, 2 ** 24, THREADS) * 2.0 ** -36).astype(f)
    c = (rng.integers(2 ** 23, 2 ** 24, THREADS) * 2.0 ** -33).astype(f)
    t = (rng.integers(1, 8, THREADS) * 2.0 ** -52).astype(f)
    return np.stack([a, b, c, t, -a, -b, -c, 0 * a])


def _two_sum(a, x):
    s = a + x
    b = s - a
    return s, (a - (s - b)) + (x - b)


def _float_sums(v, parts):
    """The device's sum of the rows of v, with two or three floats."""
    z = np.zeros(v.shape[1], np.float32)
    hi, mid, lo = z, z, z
    for x in v:
        hi, e = _two_sum(hi, x)
        s, e2 = _two_sum(mid, e)
        mid = s
        if parts == 3:
            lo = lo + e2
    return hi.astype(float) + (mid.astype(float) + lo.astype(float))


def _bound(v):
    """Eight additions round the third float, at most 2^-24 of 8 errors of 2^-24
    of 8 errors of 2^-24 of a partial sum below twice the largest term, then
    FP64 adds 256 remainders of 2^-49: below 2^-62 of the sum of magnitudes."""
    return 2.0 ** -62 * float(np.abs(v.astype(float)).sum())


def test_two_floats_would_not_do():
    v = _column(np.random.default_rng(3))
    exact = math.fsum(v.astype(float).ravel())
    assert abs(math.fsum(_float_sums(v, 3)) - exact) <= _bound(v)
    assert abs(math.fsum(_float_sums(v, 2)) - exact) > 100 * _bound(v)


@pytest.mark.gpu
@pytest.mark.parametrize('axis', [0, 1, 2])
def test_cancelling_momentum(cuda_lib, axis):
    v = _column(np.random.default_rng(3 + axis))
    u = np.zeros((3, THREADS * CELLS))
    u[axis] = v.ravel()
    sim = cuda_lib.Simulation(dict(nx=128, ny=4, nz=4, tau=0.8, geometry=0))
    sim.set_lattice(None, u)
    p = sim.diagnostics()['momentum']
    assert abs(p[axis] - math.fsum(v.astype(float).ravel())) <= _bound(v)
    assert all(p[a] == 0.0 for a in range(3) if a != axis)
