"""The cooperative launch of ibm_lbm_spread_noalloc where the context has fewer
SMs than the device reports (a partitioned GPU): a launch refused as too large
is repeated with a smaller grid. The library's host code (its object file)
against a fake CUDA runtime, on the CPU: nothing is launched."""
import ctypes
import os
import subprocess

import pytest

from paper_1704_04551_gb300 import binding, build

FAKE = r'''
#include <stddef.h>
typedef struct { unsigned x, y, z; } dim3_t;
static char scratch[16];
static void* handle = scratch;
int limit = 1 << 30, code = 720, launches = 0, last_grid = 0, last_error = 0;
void** __cudaRegisterFatBinary(void* p) { (void)p; return &handle; }
void __cudaRegisterFatBinaryEnd(void** p) { (void)p; }
void __cudaUnregisterFatBinary(void** p) { (void)p; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaLaunchKernel(void) { return 1; }
int __cudaPopCallConfiguration(void) { return 1; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int dev) { (void)attr; (void)dev; *v = 152; return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = scratch; return 0; }
int cudaMemsetAsync(void* p, int v, size_t n, void* st) { (void)p; (void)v; (void)n; (void)st; return 0; }
int cudaGetLastError(void) { int e = last_error; last_error = 0; return e; }
int cudaLaunchCooperativeKernel(const void* f, dim3_t grid, dim3_t block, void** args, size_t smem, void* st) {
  (void)f; (void)block; (void)args; (void)smem; (void)st;
  ++launches;
  last_grid = (int)grid.x;
  return last_error = last_grid > limit ? code : 0;
}
'''


@pytest.fixture(scope='module')
def lib(tmp_path_factory):
    build.build()
    d = tmp_path_factory.mktemp('fake_runtime')
    (d / 'fake.c').write_text(FAKE)
    so = str(d / 'noalloc_fake.so')
    subprocess.run(['gcc', '-shared', '-fPIC', '-O1', '-w', '-Wl,-Bsymbolic', '-o', so, str(d / 'fake.c'),
                    os.path.join(build.BUILD, 'noalloc.o'), '-lstdc++'], check=True)
    return ctypes.CDLL(so)


def _call(lib, limit, code=720):
    P = ctypes.c_void_p
    for name, v in (('limit', limit), ('code', code), ('launches', 0), ('last_error', 0)):
        ctypes.c_int.in_dll(lib, name).value = v
    fn = lib.ibm_lbm_spread_noalloc
    fn.argtypes = [P, P, ctypes.c_int64] + [ctypes.c_int32] * 4 + [ctypes.c_double, P, P]
    rc = fn(P(16), P(16), 120000, 64, 64, 64, 0, 0.0, P(16), None)
    get = lambda name: ctypes.c_int.in_dll(lib, name).value  # noqa: E731
    return rc, get('launches'), get('last_grid'), get('last_error')


def test_full_grid_where_it_fits(lib):
    assert _call(lib, 608) == (0, 1, 608, 0)


@pytest.mark.parametrize('limit', [607, 304, 76, 5, 1])
def test_smaller_grid_where_the_launch_is_refused(lib, limit):
    rc, launches, grid, error = _call(lib, limit)
    assert (rc, error) == (0, 0) and launches > 1
    assert limit / 2 < grid <= limit


def test_errors_are_reported(lib):
    assert _call(lib, 0)[0] == binding.E_CUDA  # refused at every size
    assert _call(lib, 0)[3] == 0  # (and the error cleared)
    rc, launches, _, _ = _call(lib, 0, code=719)
    assert rc == binding.E_CUDA and launches == 1
