// Coupling of few bodies in one lattice: one cluster of thread blocks per
// body (cluster_body.cuh).
#include <algorithm>

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
void launch_kind(const ClusterLaunch& Q, int n, size_t smem, cudaStream_t st) {
  switch (Q.L.geometry) {
    case GEOM_PERIODIC: k_couple_cluster<GEOM_PERIODIC, KIND><<<n * CLUSTER, CLUSTER_THREADS, smem, st>>>(Q); break;
    case GEOM_YWALLS: k_couple_cluster<GEOM_YWALLS, KIND><<<n * CLUSTER, CLUSTER_THREADS, smem, st>>>(Q); break;
    default: k_couple_cluster<GEOM_TUBE, KIND><<<n * CLUSTER, CLUSTER_THREADS, smem, st>>>(Q); break;
  }
}

}  // namespace

cudaError_t cluster_configure() {
  cudaError_t e = cudaSuccess;
#define CFG(k) if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, CLUSTER_SMEM_MAX)
  CFG((k_couple_cluster<GEOM_PERIODIC, 0>)); CFG((k_couple_cluster<GEOM_YWALLS, 0>)); CFG((k_couple_cluster<GEOM_TUBE, 0>));
  CFG((k_couple_cluster<GEOM_PERIODIC, 1>)); CFG((k_couple_cluster<GEOM_YWALLS, 1>)); CFG((k_couple_cluster<GEOM_TUBE, 1>));
#undef CFG
  return e;
}

// Cells of a block's box: what one resident wave of the launch leaves, at
// most CLUSTER_BOX_MAX (a block of a larger box adds its markers one by one
// with global atomics). 0: the fixed part alone does not fit.
int cluster_box_cells(size_t fixed_words, int n_clusters, int n_sm) {
  const int per_sm = std::max(1, (n_clusters * CLUSTER + n_sm - 1) / n_sm);
  const size_t share = std::min<size_t>(CLUSTER_SMEM_MAX, (size_t)(CLUSTER_SMEM_SM / std::min(per_sm, CLUSTER_PER_SM)) - 5 * 1024);
  if (4 * fixed_words + 12 * 1024 > share) return 0;
  return (int)std::min<size_t>(CLUSTER_BOX_MAX, (share / 4 - fixed_words) / 3);
}

void launch_couple_cluster(const LatticeDev& L, float4* g_next, uint8_t* flags_next, const MarkersDev& m,
                           BodyDev* bodies, const int* list, int n, bool membranes, int max_count,
                           const MeshDev& mesh, int4* boxes, int n_sm, bool interp, bool forces, bool spread,
                           cudaStream_t st) {
  if (n == 0) return;
  const size_t fixed = cluster_fixed_words(max_count, membranes ? mesh.nv : 0, membranes ? mesh.part_tris : 0);
  const int cap = cluster_box_cells(fixed, n, n_sm);
  const ClusterLaunch Q{L, g_next, flags_next, m, bodies, list, mesh, boxes, cap, interp, forces, spread};
  const size_t smem = 4 * fixed + 12 * (size_t)cap;
  if (membranes) launch_kind<1>(Q, n, smem, st);
  else launch_kind<0>(Q, n, smem, st);
}

}  // namespace ibm
