// Coupling of few bodies in one lattice: one cluster of thread blocks per
// body (cluster_body.cuh).
#include <algorithm>
#include <atomic>

#include "cluster_body.cuh"
#include "common.cuh"
#include "internal.h"

namespace ibm {

namespace {

struct ClusterLaunch {
  LatticeDev L;  // as the finished collision left it
  float4* g_next;
  uint8_t* flags_next;
  MarkersDev m;
  BodyDev* bodies;
  const int* list;  // body of each cluster
  MeshDev mesh;
  int4* boxes;      // [bodies][CLUSTER][2]
  int cap, interp, forces, spread;
};

template <int GEOM, int KIND>
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(CLUSTER_THREADS, CLUSTER_PER_SM)
    k_couple_cluster(const __grid_constant__ ClusterLaunch Q) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ ClusterShare S;
  const int body = Q.list[blockIdx.x / CLUSTER];
  ClusterArgs A;
  A.L = Q.L;
  A.g_next = Q.g_next;
  A.flags_next = Q.flags_next;
  A.m = Q.m;
  A.body = Q.bodies + body;
  A.mesh = Q.mesh;
  A.boxes = Q.boxes + (size_t)body * 2 * CLUSTER;
  A.cap = Q.cap;
  A.interp = Q.interp != 0;
  A.forces = Q.forces != 0;
  A.spread = Q.spread != 0;
  cluster_couple<GEOM, KIND>(A, S, smem);
}

template <int KIND>
void launch_kind(const ClusterLaunch& Q, int n, size_t smem, bool programmatic, cudaStream_t st) {
  const dim3 grid(n * CLUSTER), block(CLUSTER_THREADS);
  switch (Q.L.geometry) {
    case GEOM_PERIODIC: launch_after(k_couple_cluster<GEOM_PERIODIC, KIND>, grid, block, smem, st, programmatic, Q); break;
    case GEOM_YWALLS: launch_after(k_couple_cluster<GEOM_YWALLS, KIND>, grid, block, smem, st, programmatic, Q); break;
    default: launch_after(k_couple_cluster<GEOM_TUBE, KIND>, grid, block, smem, st, programmatic, Q); break;
  }
}

// Solid-only dynamics of few membranes (solid.cu): a cluster per body takes
// many steps in one launch. The general path launches the force kernel and a
// Verlet half step twice per step, and one block's latency decides it (66 us a
// step for a 1442-vertex cell: 2 x 42 us of forces, of which the first repeats
// the last of the step before, 2 x 5 us of FP64). Here positions, velocities
// and external forces stay in registers, each step's forces are computed once,
// and the second half of a step and the first of the next are one update. Two
// cluster barriers a step: the positions are double-buffered, so that a block
// may write the next ones while another still reads these.
constexpr int SOLID_THREADS = 512;
constexpr int SOLID_ITEMS = 5;  // coordinates a thread carries: 3 * cluster_per(nv) <= 512 * 5

struct SolidLaunch {
  MarkersDev m;
  BodyDev* bodies;
  const int* list;
  MeshDev mesh;
  double* v;           // [3][M]
  const double* fext;  // [3][M] or null
  double dt, gamma, inv_mass;
  int steps;
};

__host__ __device__ constexpr int solid_words(int nv, int nt_part) { return 3 * cluster_per(nv) + 12 * nv + 4 * nt_part; }

__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(SOLID_THREADS, 1)
    k_solid_cluster(const __grid_constant__ SolidLaunch Q) {
  using namespace cluster_detail;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ ClusterShare S;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31;
  const MarkersDev& m = Q.m;
  const size_t M = (size_t)m.M;
  BodyDev* B = Q.bodies + Q.list[blockIdx.x / CLUSTER];
  const int nv = Q.mesh.nv, per = cluster_per(nv), nt_part = Q.mesh.part_tris;
  const int c0 = min(rank * per, nv), n = min(per, nv - c0), first = B->first + c0;
  const MeshPart P = mesh_part(Q.mesh, rank);
  int* sQ = reinterpret_cast<int*>(smem);              // [3][per]
  float* pos = reinterpret_cast<float*>(sQ + 3 * per);  // [2][6][nv]
  float* sN = pos + 12 * nv;                           // [3][nt_part]
  float* sA = sN + 3 * nt_part;                        // [nt_part]
  const int o[3] = {m.cell[B->first], m.cell[M + B->first], m.cell[2 * M + B->first]};
  const MembraneModuli Km{B->kBT_p, B->k_b, B->k_l, B->k_g, B->k_v};
  float q_prev = B->qmax;
  const double h = 0.5 * Q.dt, damp = 1.0 / (1.0 + 0.5 * Q.gamma * Q.dt);
  // item i of this thread: coordinate a of own vertex j
  double X[SOLID_ITEMS], v[SOLID_ITEMS], fe[SOLID_ITEMS];
  float F[SOLID_ITEMS];
#pragma unroll
  for (int t = 0; t < SOLID_ITEMS; ++t) {
    const int i = tid + t * SOLID_THREADS;
    X[t] = v[t] = fe[t] = 0.0;
    F[t] = 0.f;
    if (i >= 3 * n) continue;
    const int a = i / n;
    const size_t k = a * M + first + (i - a * n);
    X[t] = m.X[k];
    v[t] = Q.v[k];
    fe[t] = Q.fext ? Q.fext[k] * Q.inv_mass : 0.0;
  }
  for (int i = tid; i < 3 * per; i += SOLID_THREADS) sQ[i] = 0;
  if (tid == 0) S.part_sum = BodySums{};
  if (tid < CLUSTER) S.qmax[tid] = 0u;
  if (tid == 0) S.fmax_s = S.redo_max = 0u;
  cl.sync();  // every block has started and has read the origin
  // s = -1: forces at the start; step s: Verlet update to new positions, their forces
  for (int s = -1; s < Q.steps; ++s) {
    float* sI = pos + ((s & 1) ? 6 * nv : 0);
    float* sR = sI + 3 * nv;
#pragma unroll
    for (int t = 0; t < SOLID_ITEMS; ++t) {
      const int i = tid + t * SOLID_THREADS;
      if (i >= 3 * n) continue;
      const int a = i / n, j = i - a * n;
      if (s >= 0) {
        const double acc = fma((double)F[t], Q.inv_mass, fe[t]);
        if (s > 0) v[t] = fma(h, acc, v[t]) * damp;  // second half of step s - 1
        v[t] = fma(h, fma(-Q.gamma, v[t], acc), v[t]);
        X[t] = fma(Q.dt, v[t], X[t]);
      }
      int c;
      float f;
      split_coord(X[t], c, f);
      const float fc = (float)(c - o[a]);
#pragma unroll
      for (int r = 0; r < CLUSTER; ++r) {
        cl.map_shared_rank(sI, r)[a * nv + c0 + j] = fc;
        cl.map_shared_rank(sR, r)[a * nv + c0 + j] = f;
      }
    }
    cl.sync();  // positions complete; every block is done with the last sums
    float unit;
    float qmax = cluster_membrane<SOLID_THREADS>(S, MembraneArrays{sI, sR, sN, sA, sQ, nv, nt_part, per, c0, n}, P,
                                                 Q.mesh, Km, q_prev, unit);
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, w));
    if (lane == 0) atomicMax(&S.fmax_s, __float_as_uint(qmax));  // non-negative floats order as their bits
    __syncthreads();  // the sums and the largest contribution are complete
    const float qb = __uint_as_float(S.fmax_s);
    q_prev = isfinite(qb) ? qb : 0.f;  // this block's scale: its own largest contribution
#pragma unroll
    for (int t = 0; t < SOLID_ITEMS; ++t) {
      const int i = tid + t * SOLID_THREADS;
      if (i >= 3 * n) continue;
      const int a = i / n, j = i - a * n, q = a * per + j;
      F[t] = unit > 0.f ? (float)sQ[q] * unit : __int_as_float(sQ[q]);
      sQ[q] = 0;
    }
    __syncthreads();  // (all have read the maximum)
    if (tid == 0) S.fmax_s = 0u;
    if (tid == 0) S.part_sum = BodySums{};
  }
  if (tid == 0) cl.map_shared_rank(&S.qmax[0], 0)[rank] = __float_as_uint(q_prev);
#pragma unroll
  for (int t = 0; t < SOLID_ITEMS; ++t) {
    const int i = tid + t * SOLID_THREADS;
    if (i >= 3 * n) continue;
    const int a = i / n, j = i - a * n;
    const size_t k = a * M + first + j;
    if (Q.steps > 0) v[t] = fma(h, fma((double)F[t], Q.inv_mass, fe[t]), v[t]) * damp;
    Q.v[k] = v[t];
    m.X[k] = X[t];
    cache_coord(m, k, X[t]);
    reinterpret_cast<float*>(m.F + first + j)[a] = F[t];
  }
  cl.sync();
  if (rank == 0 && tid == 0) {
    float q = 0.f;
    for (int r = 0; r < CLUSTER; ++r) q = fmaxf(q, __uint_as_float(S.qmax[r]));
    B->qmax = q;
  }
}

}  // namespace

cudaError_t cluster_configure() {
  cudaError_t e = cudaSuccess;
#define CFG(k) if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, CLUSTER_SMEM_MAX)
  CFG((k_couple_cluster<GEOM_PERIODIC, 0>)); CFG((k_couple_cluster<GEOM_YWALLS, 0>)); CFG((k_couple_cluster<GEOM_TUBE, 0>));
  CFG((k_couple_cluster<GEOM_PERIODIC, 1>)); CFG((k_couple_cluster<GEOM_YWALLS, 1>)); CFG((k_couple_cluster<GEOM_TUBE, 1>));
  CFG(k_solid_cluster);
#undef CFG
  return e;
}

bool solid_cluster_fits(const MeshDev& mesh) {
  return 3 * cluster_per(mesh.nv) <= SOLID_THREADS * SOLID_ITEMS &&
         4 * (size_t)solid_words(mesh.nv, mesh.part_tris) <= (size_t)CLUSTER_SMEM_MAX;
}

void launch_solid_cluster(const MarkersDev& m, BodyDev* bodies, const int* list, int n, const MeshDev& mesh, double* v,
                          const double* fext, double dt, double gamma, double mass, int steps, cudaStream_t st) {
  const SolidLaunch Q{m, bodies, list, mesh, v, fext, dt, gamma, 1.0 / mass, steps};
  k_solid_cluster<<<n * CLUSTER, SOLID_THREADS, 4 * (size_t)solid_words(mesh.nv, mesh.part_tris), st>>>(Q);
}

// Clusters the device holds at once with `per_sm` blocks on an SM. Fewer than
// its SMs give room for: a cluster's blocks lie in one GPC, and GPCs are not
// all of a size (152 SMs: 15 clusters of one block an SM, 36 of two, not 19
// and 38; with one block an SM 16 to 19 bodies took two waves, 72 us a step
// instead of 45 with two for membranes of 642 vertices at 72^3).
// (Asked once per device: ~8 us, and every handle needs both.)
cudaError_t cluster_capacity(int per_sm, int* out) {
  constexpr int DEVICES = 64;
  static std::atomic<int> known[2][DEVICES];  // 0: not asked yet
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::atomic<int>* slot = dev < DEVICES ? &known[per_sm == 1 ? 0 : 1][dev] : nullptr;
  if (slot && (*out = slot->load()) > 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CLUSTER);
  cfg.blockDim = dim3(CLUSTER_THREADS);
  cfg.dynamicSmemBytes = per_sm == 1 ? (size_t)CLUSTER_SMEM_MAX : (size_t)CLUSTER_SHARE;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CLUSTER;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(out, k_couple_cluster<GEOM_TUBE, 1>, &cfg);
  if (e == cudaSuccess && slot) slot->store(*out);
  return e;
}

// Cells of a block's box: what `per_sm` blocks on an SM leave, at most
// CLUSTER_BOX_MAX (a block of a larger box adds its markers one by one with
// global atomics). 0: the fixed part alone does not fit.
int cluster_box_cells(size_t fixed_words, int per_sm) {
  const size_t share = per_sm == 1 ? (size_t)CLUSTER_SMEM_MAX : (size_t)CLUSTER_SHARE;
  if (4 * fixed_words + 12 * 1024 > share) return 0;
  return (int)std::min<size_t>(CLUSTER_BOX_MAX, (share / 4 - fixed_words) / 3) & ~3;  // (cleared 16 bytes at a time)
}

void launch_couple_cluster(const LatticeDev& L, float4* g_next, uint8_t* flags_next, const MarkersDev& m,
                           BodyDev* bodies, const int* list, int n, bool membranes, int max_count,
                           const MeshDev& mesh, int4* boxes, int per_sm, bool interp, bool forces, bool spread,
                           bool programmatic, cudaStream_t st) {
  if (n == 0) return;
  const size_t fixed = cluster_fixed_words(max_count, membranes ? mesh.nv : 0, membranes ? mesh.part_tris : 0);
  const int cap = cluster_box_cells(fixed, per_sm);
  const ClusterLaunch Q{L, g_next, flags_next, m, bodies, list, mesh, boxes, cap, interp, forces, spread};
  const size_t smem = 4 * fixed + 12 * (size_t)cap;
  if (membranes) launch_kind<1>(Q, n, smem, programmatic, st);
  else launch_kind<0>(Q, n, smem, programmatic, st);
}

}  // namespace ibm
