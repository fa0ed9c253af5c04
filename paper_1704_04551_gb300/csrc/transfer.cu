// Immersed-boundary transfer kernels of one lattice (Sec. 2.3 of
// arXiv:1704.04551): spreading (Eq. ibmForceSpread) and interpolation with
// advection (Eq. ibmVelocityInterpret), one thread block per marker group;
// the group bodies and their design notes are in transfer_group.cuh.
#include "common.cuh"
#include "internal.h"
#include "transfer_group.cuh"

namespace ibm {

// Stencil cache from the positions (after set_markers).
__global__ void k_stencil_cache(MarkersDev m) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m.M) return;
  const size_t M = (size_t)m.M;
  for (int a = 0; a < 3; ++a) cache_coord(m, a * M + k, m.X[a * M + k]);
}

template <int GEOM>
__global__ void __launch_bounds__(XFER_THREADS, 2) k_spread(LatticeDev L, MarkersDev m, const MarkerGroup* groups,
                                                            int4* boxes) {
  extern __shared__ __align__(16) unsigned char smem[];  // fixed-point box, marker records
  spread_group<GEOM>(L, m, groups[blockIdx.x], boxes + 2 * blockIdx.x, smem);
}

template <int GEOM>
__global__ void __launch_bounds__(XFER_THREADS, 2) k_interpolate(LatticeDev L, MarkersDev m,
                                                                 const MarkerGroup* groups, const int4* boxes) {
  extern __shared__ __align__(16) unsigned char smem[];  // velocity box, marker records
  interpolate_group<GEOM>(L, m, groups[blockIdx.x], boxes + 2 * blockIdx.x, smem);
}

// The same for launches of fewer than LANE_MAX_GROUPS groups (four lanes
// per marker).
template <int GEOM>
__global__ void __launch_bounds__(LANE_THREADS, 1) k_spread_lanes(LatticeDev L, MarkersDev m,
                                                                 const MarkerGroup* groups, int4* boxes) {
  extern __shared__ __align__(16) int ibox[];  // fixed-point box
  spread_group_lanes<GEOM>(L, m, groups[blockIdx.x], boxes + 2 * blockIdx.x, ibox);
}

template <int GEOM>
__global__ void __launch_bounds__(LANE_THREADS, 1) k_interpolate_lanes(LatticeDev L, MarkersDev m,
                                                                      const MarkerGroup* groups, const int4* boxes) {
  extern __shared__ __align__(16) unsigned char smem[];  // velocity box
  interpolate_group_lanes<GEOM>(L, m, groups[blockIdx.x], boxes + 2 * blockIdx.x, smem);
}

// Tracers (markers outside every body) carry no force in a step: their stencils
// are marked where the collision is to write velocities, and they move. They
// may lie anywhere, so there is no box: four lanes per marker read straight
// from the lattice, 64 consecutive bytes per stencil row, with the arithmetic
// of interpolate_group_lanes (the same bits). Bound by the L2 reads, 1 KB a
// marker. As groups of the body kernels, whose boxes such tracers do not fit,
// 150,000 of them in a 131x96x110 box took 121 us to move (64 loads in a chain
// of 16, and as many stores that cleared a force density never spread) and 63
// us to mark.
constexpr int TRACER_THREADS = 256, TRACER_PARTS = 4;  // blocks per group, 64 markers each
static_assert(TRACER_GROUP == TRACER_THREADS / 4 * TRACER_PARTS, "tracer blocks cover a group");

template <int GEOM>
__global__ void __launch_bounds__(TRACER_THREADS, 4) k_tracers_move(LatticeDev L, MarkersDev m, const MarkerGroup* groups) {
  const MarkerGroup G = groups[blockIdx.x / TRACER_PARTS];
  const int a = threadIdx.x & 3, j = (blockIdx.x % TRACER_PARTS) * (TRACER_THREADS / 4) + (threadIdx.x >> 2);
  const bool active = j < G.count;
  const size_t M = (size_t)m.M;
  const int k = G.first + (active ? j : 0);
  const size_t off = (size_t)(a < 3 ? a : 0) * M + k;
  RawStencil rs;
  load_raw(m, k, rs);
  const double Xo = m.X[off];
  const int x = wrapi(rs.c[0] - 1 + a, L.nx);
  const float wxa = axis_weight(rs.f[0], a);
  float wy[4], wz[4];
  axis_weights(rs.f[1], wy);
  axis_weights(rs.f[2], wz);
  float ux = 0.f, uy = 0.f, uz = 0.f;
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // eight loads in flight
    float4 v[8];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        int y = rs.c[1] - 1 + b, z = rs.c[2] - 1 + 2 * h + c;
        const bool fluid = fluid_row<GEOM>(L, y, z);
        v[4 * c + b] = fluid ? __ldg(L.uw + (size_t)L.nx * (y + L.ny * z) + x) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float wyz = wy[b] * wz[2 * h + c];
        ux = fmaf(wyz, v[4 * c + b].x, ux);
        uy = fmaf(wyz, v[4 * c + b].y, uy);
        uz = fmaf(wyz, v[4 * c + b].z, uz);
      }
  }
  ux *= wxa;
  uy *= wxa;
  uz *= wxa;
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    ux += __shfl_xor_sync(0xffffffffu, ux, o);
    uy += __shfl_xor_sync(0xffffffffu, uy, o);
    uz += __shfl_xor_sync(0xffffffffu, uz, o);
  }
  if (!active) return;
  if (a == 0) m.U[k] = make_float4(ux, uy, uz, 0.f);
  if (a < 3) {
    const double Xn = Xo + (double)(a == 0 ? ux : (a == 1 ? uy : uz));
    m.X[off] = Xn;
    cache_coord(m, off, Xn);
  }
}

template <int GEOM>
__global__ void k_tracers_mark(LatticeDev L, MarkersDev m, const MarkerGroup* groups) {
  const MarkerGroup G = groups[blockIdx.x];
  for (int j0 = 0; j0 + (int)(threadIdx.x & ~31u) < G.count; j0 += blockDim.x) {  // whole warps (shuffles)
    const int j = j0 + threadIdx.x;
    const bool active = j < G.count;
    const int k = G.first + (active ? j : 0);
    const size_t M = (size_t)m.M;
    mark_tiles<GEOM>(L, m.cell[k] - 1, m.cell[M + k] - 1, m.cell[2 * M + k] - 1, active);
  }
}

void launch_tracers_move(const LatticeDev& L, const MarkersDev& m, const MarkerGroup* groups, int n, cudaStream_t st) {
  if (n == 0) return;
  const int grid = n * TRACER_PARTS;
  switch (L.geometry) {
    case GEOM_PERIODIC: k_tracers_move<GEOM_PERIODIC><<<grid, TRACER_THREADS, 0, st>>>(L, m, groups); break;
    case GEOM_YWALLS: k_tracers_move<GEOM_YWALLS><<<grid, TRACER_THREADS, 0, st>>>(L, m, groups); break;
    default: k_tracers_move<GEOM_TUBE><<<grid, TRACER_THREADS, 0, st>>>(L, m, groups); break;
  }
}

void launch_tracers_mark(const LatticeDev& L, const MarkersDev& m, const MarkerGroup* groups, int n, cudaStream_t st) {
  if (n == 0) return;
  switch (L.geometry) {
    case GEOM_PERIODIC: k_tracers_mark<GEOM_PERIODIC><<<n, TRACER_GROUP, 0, st>>>(L, m, groups); break;
    case GEOM_YWALLS: k_tracers_mark<GEOM_YWALLS><<<n, TRACER_GROUP, 0, st>>>(L, m, groups); break;
    default: k_tracers_mark<GEOM_TUBE><<<n, TRACER_GROUP, 0, st>>>(L, m, groups); break;
  }
}

cudaError_t transfer_configure() {
  cudaError_t e = cudaSuccess;
#define CFG(k, smem) if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
  CFG(k_spread<GEOM_PERIODIC>, SPREAD_SMEM); CFG(k_spread<GEOM_YWALLS>, SPREAD_SMEM); CFG(k_spread<GEOM_TUBE>, SPREAD_SMEM);
  CFG(k_interpolate<GEOM_PERIODIC>, INTERP_SMEM); CFG(k_interpolate<GEOM_YWALLS>, INTERP_SMEM);
  CFG(k_interpolate<GEOM_TUBE>, INTERP_SMEM);
  CFG(k_spread_lanes<GEOM_PERIODIC>, SPREAD_LANES_SMEM); CFG(k_spread_lanes<GEOM_YWALLS>, SPREAD_LANES_SMEM);
  CFG(k_spread_lanes<GEOM_TUBE>, SPREAD_LANES_SMEM);
  CFG(k_interpolate_lanes<GEOM_PERIODIC>, INTERP_SMEM); CFG(k_interpolate_lanes<GEOM_YWALLS>, INTERP_SMEM);
  CFG(k_interpolate_lanes<GEOM_TUBE>, INTERP_SMEM);
#undef CFG
  return e;
}

// (x, y, z, -) float4 [M] -> FP64 [3][M] (marker velocities and forces for
// the API).
__global__ void k_expand_xyz(const float4* in, double* out, int M) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= M) return;
  const float4 v = in[k];
  out[k] = v.x;
  out[(size_t)M + k] = v.y;
  out[2 * (size_t)M + k] = v.z;
}

void launch_expand_xyz(const float4* in, double* out, int M, cudaStream_t st) {
  if (M > 0) k_expand_xyz<<<(M + 255) / 256, 256, 0, st>>>(in, out, M);
}

void launch_stencil_cache(const MarkersDev& m, cudaStream_t st) {
  if (m.M == 0) return;
  k_stencil_cache<<<(m.M + 255) / 256, 256, 0, st>>>(m);
}

void launch_spread(const LatticeDev& L, const MarkersDev& m, const MarkerGroup* groups, int n_groups, int4* boxes,
                   cudaStream_t st) {
  if (m.M == 0 || n_groups == 0) return;
  if (n_groups < LANE_MAX_GROUPS) {
    const size_t smem = SPREAD_LANES_SMEM;
    switch (L.geometry) {
      case GEOM_PERIODIC: k_spread_lanes<GEOM_PERIODIC><<<n_groups, LANE_THREADS, smem, st>>>(L, m, groups, boxes); break;
      case GEOM_YWALLS: k_spread_lanes<GEOM_YWALLS><<<n_groups, LANE_THREADS, smem, st>>>(L, m, groups, boxes); break;
      default: k_spread_lanes<GEOM_TUBE><<<n_groups, LANE_THREADS, smem, st>>>(L, m, groups, boxes); break;
    }
    return;
  }
  const size_t smem = SPREAD_SMEM;
  switch (L.geometry) {
    case GEOM_PERIODIC: k_spread<GEOM_PERIODIC><<<n_groups, XFER_THREADS, smem, st>>>(L, m, groups, boxes); break;
    case GEOM_YWALLS: k_spread<GEOM_YWALLS><<<n_groups, XFER_THREADS, smem, st>>>(L, m, groups, boxes); break;
    default: k_spread<GEOM_TUBE><<<n_groups, XFER_THREADS, smem, st>>>(L, m, groups, boxes); break;
  }
}

void launch_interpolate(const LatticeDev& L, const MarkersDev& m, const MarkerGroup* groups, int n_groups,
                        const int4* boxes, cudaStream_t st) {
  if (m.M == 0 || n_groups == 0) return;
  const size_t smem = INTERP_SMEM;
  if (n_groups < LANE_MAX_GROUPS) {
    switch (L.geometry) {
      case GEOM_PERIODIC:
        k_interpolate_lanes<GEOM_PERIODIC><<<n_groups, LANE_THREADS, smem, st>>>(L, m, groups, boxes);
        break;
      case GEOM_YWALLS: k_interpolate_lanes<GEOM_YWALLS><<<n_groups, LANE_THREADS, smem, st>>>(L, m, groups, boxes); break;
      default: k_interpolate_lanes<GEOM_TUBE><<<n_groups, LANE_THREADS, smem, st>>>(L, m, groups, boxes); break;
    }
    return;
  }
  switch (L.geometry) {
    case GEOM_PERIODIC: k_interpolate<GEOM_PERIODIC><<<n_groups, XFER_THREADS, smem, st>>>(L, m, groups, boxes); break;
    case GEOM_YWALLS: k_interpolate<GEOM_YWALLS><<<n_groups, XFER_THREADS, smem, st>>>(L, m, groups, boxes); break;
    default: k_interpolate<GEOM_TUBE><<<n_groups, XFER_THREADS, smem, st>>>(L, m, groups, boxes); break;
  }
}

}  // namespace ibm
