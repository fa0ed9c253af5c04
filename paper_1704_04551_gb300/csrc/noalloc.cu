// Force spreading without device allocation (ibm_lbm_spread_noalloc).
//
// For callers that cannot call cudaMalloc (a framework that has reserved the
// GPU's memory for its own pool, a loop that may not pay allocation cost):
// the accumulator lives in a file-scope device array of fixed size instead
// of memory the library allocates. The operation is the spreading of Eq.
// ibmForceSpread with the 4-point cosine delta of Eq. deltaPhiSimple, the
// same as the SPREAD stage of a handle.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/ibm_lbm.h"
#include "common.cuh"

namespace ibm {
namespace {

// One accumulator per device, shared by every call on that device. In host
// code this name is only a stand-in for the device array; its device address
// comes from cudaGetSymbolAddress below.
static __device__ __align__(256) float4 g_noalloc_scratch[IBM_LBM_NOALLOC_MAX_CELLS];

// Device address of the accumulator in the current context. Looked up on
// every call (a host-side table lookup once the module is loaded) rather than
// cached: if the caller resets the device, the module is loaded again and the
// array may move, and a cached address would then point at freed memory.
cudaError_t scratch_address(float4** out) {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess) return e;
  *out = static_cast<float4*>(p);
  return cudaSuccess;
}

struct Grid {
  int nx, ny, nz, N, geometry;
  float yc, zc, R2;
};

__device__ __forceinline__ bool grid_solid(const Grid& G, int y, int z) {
  if (G.geometry == GEOM_YWALLS) return (unsigned)y >= (unsigned)G.ny;
  if (G.geometry == GEOM_TUBE) {
    if ((unsigned)y >= (unsigned)G.ny || (unsigned)z >= (unsigned)G.nz) return true;
    const float dy = (float)y - G.yc, dz = (float)z - G.zc;
    return dy * dy + dz * dz > G.R2;
  }
  return false;
}

// One cooperative launch: clears the accumulator, spreads, writes g out, with
// a grid barrier between the parts. (As a memset and two kernels, a call of
// one body's markers on a 48x40x36 lattice took 22 us, most of it launches and
// one thread's walk through its marker's 64 nodes; a 101x97x103 lattice with
// 120,000 markers took 63 us, 49 of them the spreading.) Sixteen lanes share a
// marker: lane q < 3 splits coordinate q and rounds force component q (FP64
// conversions run at 2 lanes a cycle on an SM: once per marker), lanes 0..11
// evaluate one of the twelve weights each; then four lanes add the four nodes
// of an x row, 64 consecutive bytes, and the lane groups take four rows a pass
// (one lane per row, each atomic a sector of its own, took 55 us on the second
// lattice above).
constexpr int SPREAD_THREADS = 256;
constexpr int SPREAD_BLOCKS_PER_SM = 4;
constexpr int SPREAD_LANES = 16;

__global__ void __launch_bounds__(SPREAD_THREADS, SPREAD_BLOCKS_PER_SM)
    k_spread_noalloc(Grid G, const double* __restrict__ X, const double* __restrict__ F, int M, float4* acc, double* g) {
  const cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  const unsigned tid = blockIdx.x * (unsigned)SPREAD_THREADS + threadIdx.x;
  const unsigned threads = gridDim.x * (unsigned)SPREAD_THREADS;
  for (unsigned i = tid; i < (unsigned)G.N; i += threads) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  grid.sync();
  const int lane = threadIdx.x & (SPREAD_LANES - 1);
  const unsigned group = tid / SPREAD_LANES, groups = threads / SPREAD_LANES;
  // whole warps iterate together (shuffles)
  const unsigned warp_group = group & ~1u;
  for (unsigned k0 = 0; k0 + warp_group < (unsigned)M; k0 += groups) {
    const unsigned k = k0 + group;
    const bool active = k < (unsigned)M;
    // Positions come straight from device memory, unchecked by the host: a
    // marker that is not finite or lies at |x| >= 2^30 (the bound the handle's
    // set_markers enforces) is skipped, so that no index below overflows.
    int cell = 0;
    float frac = 0.f, force = 0.f;
    bool bad = !active;
    if (active && lane < 3) {
      const size_t off = (size_t)lane * (size_t)M + k;
      const double x = X[off];
      bad = ((__double2hiint(x) >> 20) & 0x7ff) >= 1023 + 30;  // exponent of 2^30 and above, infinities, NaN
      if (!bad) split_coord(x, cell, frac);
      force = (float)F[off];
    }
    const unsigned votes = __ballot_sync(0xffffffffu, bad);
    const bool skip = ((votes >> (threadIdx.x & 16u)) & 7u) != 0u;
    constexpr unsigned ALL = 0xffffffffu;
    // weight lane & 3 of axis lane / 4
    const float f = __shfl_sync(ALL, frac, min(lane >> 2, 2), SPREAD_LANES);
    const float weight = 0.25f * (1.0f + cospif(0.5f * ((float)((lane & 3) - 1) - f)));
    const int a = lane & 3, b = lane >> 2;
    const float wx = __shfl_sync(ALL, weight, a, SPREAD_LANES), wy = __shfl_sync(ALL, weight, 4 + b, SPREAD_LANES);
    float wz[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) wz[c] = __shfl_sync(ALL, weight, 8 + c, SPREAD_LANES);
    const int bx = __shfl_sync(ALL, cell, 0, SPREAD_LANES) - 1 + a;
    int y = __shfl_sync(ALL, cell, 1, SPREAD_LANES) - 1 + b;
    const int bz = __shfl_sync(ALL, cell, 2, SPREAD_LANES) - 1;
    const float fx = __shfl_sync(ALL, force, 0, SPREAD_LANES), fy = __shfl_sync(ALL, force, 1, SPREAD_LANES),
                fz = __shfl_sync(ALL, force, 2, SPREAD_LANES);
    if (skip) continue;
    const int x = wrapi(bx, G.nx);
    if (G.geometry == GEOM_PERIODIC) y = wrapi(y, G.ny);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      int z = bz + c;
      if (G.geometry != GEOM_TUBE) z = wrapi(z, G.nz);
      if (grid_solid(G, y, z)) continue;
      const float w = wx * (wy * wz[c]);
      atomicAdd(acc + G.nx * (y + G.ny * z) + x, make_float4(fx * w, fy * w, fz * w, 0.f));
    }
  }
  grid.sync();
  const size_t N = (size_t)G.N;
  for (unsigned i = tid; i < (unsigned)G.N; i += threads) {
    const float4 v = __ldcg(acc + i);
    g[i] = v.x;
    g[N + i] = v.y;
    g[2 * N + i] = v.z;
  }
}

}  // namespace
}  // namespace ibm

namespace {
int spread_noalloc(const double* X, const double* F, int64_t n_markers, int32_t nx, int32_t ny, int32_t nz,
                   int32_t geometry, double tube_radius, double* g, void* stream) {
  using namespace ibm;
  const long long N = (long long)nx * ny * nz;
  if (nx < 4 || ny < 4 || nz < 4 || N > IBM_LBM_NOALLOC_MAX_CELLS) return IBM_LBM_E_ARG;
  if (n_markers < 0 || n_markers >= (1LL << 31) || (n_markers > 0 && (!X || !F)) || !g) return IBM_LBM_E_ARG;
  if (geometry < 0 || geometry > 2 || (geometry == 2 && !(tube_radius > 0))) return IBM_LBM_E_ARG;
  float4* acc = nullptr;
  if (scratch_address(&acc) != cudaSuccess) {
    cudaGetLastError();
    return IBM_LBM_E_CUDA;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n_markers == 0) {  // (100^3: 16.5 us with the accumulator cleared and read)
    if (cudaMemsetAsync(g, 0, 3 * sizeof(double) * (size_t)N, st) == cudaSuccess) return IBM_LBM_OK;
    cudaGetLastError();
    return IBM_LBM_E_CUDA;
  }
  Grid G{nx, ny, nz, (int)N, geometry, 0.5f * (float)(ny - 1), 0.5f * (float)(nz - 1),
         (float)(tube_radius * tube_radius)};
  int M = (int)n_markers, dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return IBM_LBM_E_CUDA;
  }
  // all blocks resident at once (grid barrier); fewer where there is little to do
  const long long work = std::max((N + 1) / 2, (long long)M * SPREAD_LANES);
  unsigned blocks = (unsigned)std::min<long long>((work + SPREAD_THREADS - 1) / SPREAD_THREADS,
                                                  (long long)sms * SPREAD_BLOCKS_PER_SM);
  void* args[] = {&G, &X, &F, &M, &acc, &g};
  // (a context may have fewer SMs than the device; the kernel's loops cover any grid)
  for (;; blocks = (blocks + 1) / 2) {
    const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_spread_noalloc, dim3(blocks),
                                                      dim3(SPREAD_THREADS), args, 0, st);
    if (e == cudaSuccess) return IBM_LBM_OK;
    cudaGetLastError();
    if (e != cudaErrorCooperativeLaunchTooLarge || blocks == 1) return IBM_LBM_E_CUDA;
  }
}
}  // namespace

// No C++ exception crosses the C ABI (there is no handle to carry a message).
extern "C" int ibm_lbm_spread_noalloc(const double* X, const double* F, int64_t n_markers, int32_t nx, int32_t ny,
                                      int32_t nz, int32_t geometry, double tube_radius, double* g,
                                      void* stream) {
  try {
    return spread_noalloc(X, F, n_markers, nx, ny, nz, geometry, tube_radius, g, stream);
  } catch (...) {
    return IBM_LBM_E_ARG;
  }
}
