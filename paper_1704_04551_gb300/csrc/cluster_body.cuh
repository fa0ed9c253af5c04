// Coupling of few bodies: one cluster of CLUSTER thread blocks per body does
// the interpolation and advection of step n, the body's forces, and the
// spreading of step n+1 (Secs. 2.2 and 2.3 of arXiv:1704.04551), for rigid
// bodies (penalty tether or direct forcing) and membranes. Shared by the
// single-lattice kernels (cluster.cu) and the batched serving kernels
// (serve.cu).
//
// A case with few bodies is bound by the latency of one body's chain of
// passes, and most of all by FP64: an SM does 2 FP64 lanes a cycle here, so
// the advection, the tether forces and the Newton-Euler update of one
// 812-marker body took ~20 us on one SM, beside 15 us for a gather and 21 us
// for a scatter by a single block. Here each block of the cluster takes an
// eighth of the body's markers on an SM of its own, and the three kernels
// are one.
//
// Block r of a cluster owns markers [r per, (r + 1) per), per = count / 8
// rounded up. It
//   1. gathers its markers' velocities straight from the lattice (L1/L2; four
//      lanes per marker, 16 independent loads per lane: no staging pass) and
//      advects them in FP64;
//   2. computes their forces: rigid markers alone; membrane vertices from
//      the whole body's positions, which the blocks write to one another
//      through distributed shared memory, with the edges and triangles that
//      touch its own vertices (the template is partitioned on the host);
//   3. scatters them, fixed point with one scale for the body, into a box of
//      its own in shared memory; then the rows of the body's box are dealt
//      out to the blocks, each of which adds up the blocks' sums of a cell
//      (integers: the same bits as spread_group's) and adds them to the
//      lattice with one float4 atomic per cell and body.
// The force density and tile flags the finished collision consumed are cleared
// while the blocks wait for one another. A ninth warp of block 0 does the
// Newton-Euler update beside the scatter and the flush (direct forcing: in
// every block before the scatter, since the markers go to the new pose).
//
// The step's tile flags are double-buffered like the force density: a block
// clears those of the finished step and sets those of the next in the other
// buffer, so that no memset runs between two steps.
#pragma once
#include <cooperative_groups.h>

#include "common.cuh"
#include "forces_body.cuh"
#include "transfer_group.cuh"

namespace ibm {

constexpr int CLUSTER_WORKERS = 224;     // threads that work on markers (7 warps; an eighth does the rest)
constexpr int CLUSTER_THREADS = CLUSTER_WORKERS + 32;
constexpr int CLUSTER_MAX_COUNT = 4096;  // markers per body
constexpr int CLUSTER_BOX_MAX = 12288;   // cells of a block's box
constexpr int CLUSTER_UNION_MAX = 1 << 18;  // cells of a body's box (its blocks' boxes together)
constexpr int CLUSTER_CLEAR_AHEAD = 1024;   // cells a block's last warp clears while the others gather
constexpr int CLUSTER_PER_SM = 2;        // resident blocks the registers are sized for
constexpr int CLUSTER_SMEM_SM = 227 * 1024, CLUSTER_SMEM_MAX = 220 * 1024;
// dynamic shared memory of a block at CLUSTER_PER_SM blocks
constexpr int CLUSTER_SHARE = CLUSTER_SMEM_SM / CLUSTER_PER_SM - 5 * 1024;

// Shared memory of one block, in this order (floats / ints, 16-byte aligned
// sections): own markers' cells [3][per], fractions [3][per], forces [3][per]
// (membranes: fixed-point sums); for membranes positions of the whole body
// [6][nv], normals [3][nt_part], areas [nt_part]; then the box [3][cap].
__host__ __device__ constexpr int cluster_per(int count) { return (count + CLUSTER - 1) / CLUSTER; }
__host__ __device__ constexpr int cluster_fixed_words(int count, int nv, int nt_part) {
  return (9 * cluster_per(count) + 6 * nv + 4 * nt_part + 3) / 4 * 4;
}

struct RigidPrep {
  double R0, R1, R2, wb, g, inv_I, inv_m, V, C;
};

// What the blocks of a cluster tell one another.
struct ClusterShare {
  int4 lo[CLUSTER], dims[CLUSTER];  // their boxes (dims.w: the markers fit and were scattered there)
  int4 old_lo[CLUSTER], old_dims[CLUSTER];  // the boxes of the step before
  unsigned fmax[CLUSTER];           // their largest force component
  double sum[CLUSTER][6];           // partial force and torque, or area and volume
  unsigned qmax[CLUSTER];           // largest membrane force contribution
  int lo_s[3], hi_s[3];             // own bounds
  unsigned fmax_s, redo_max;
  RigidPrep prep[3];                // per component (rigid_prepare)
  double quat[4];
  double total[6];                  // force and torque of all blocks
  double pose[12];                  // C, q (4), V; direct forcing
  double part[CLUSTER_WORKERS / 32][6];
  BodySums part_sum;                // this block's area and volume
};

// Arguments of one body's coupling: the lattice as the finished collision
// left it (L.g and L.flags are consumed), the buffers of the next collision.
struct ClusterArgs {
  LatticeDev L;
  float4* g_next;
  uint8_t* flags_next;
  MarkersDev m;
  BodyDev* body;
  MeshDev mesh;
  int4* boxes;   // [CLUSTER][2] of this body: the boxes spread into last
  int cap;       // cells of the shared-memory box
  bool interp;   // interpolation and advection of the finished step
  bool forces;   // forces of the next step
  bool spread;   // and their spreading
};

namespace cluster_detail {

namespace cg = cooperative_groups;

// Newton-Euler step of a rigid body (forces_body.cuh: rigid_update) by one
// warp: lane a < 3 carries component a, so that the dependent FP64 chain (the
// pipe's latency, ~8 us when one thread did all of it between two cluster
// barriers) is a third as long. What the old state alone decides is computed
// ahead (rigid_prepare, while the other warps gather): column a of R, the
// body-frame spin and its gyroscopic term.
__device__ __forceinline__ void rigid_prepare(const BodyDev* B, ClusterShare& S) {
  const int lane = threadIdx.x & 31, a = lane < 3 ? lane : lane % 3, b = (a + 1) % 3, c = (a + 2) % 3;
  constexpr unsigned ALL = 0xffffffffu;
  const double w = B->quat[0], x = B->quat[1], y = B->quat[2], z = B->quat[3];
  double R0, R1, R2;  // R[k][a]
  if (a == 0) { R0 = 1 - 2 * (y * y + z * z); R1 = 2 * (x * y + w * z); R2 = 2 * (x * z - w * y); }
  else if (a == 1) { R0 = 2 * (x * y - w * z); R1 = 1 - 2 * (x * x + z * z); R2 = 2 * (y * z + w * x); }
  else { R0 = 2 * (x * z + w * y); R1 = 2 * (y * z - w * x); R2 = 1 - 2 * (x * x + y * y); }
  const double wb = R0 * B->omega[0] + R1 * B->omega[1] + R2 * B->omega[2];
  const double Iw = B->inertia[a] * wb;
  const double g = __shfl_sync(ALL, wb, b) * __shfl_sync(ALL, Iw, c) - __shfl_sync(ALL, wb, c) * __shfl_sync(ALL, Iw, b);
  if (lane < 3) {
    RigidPrep& P = S.prep[a];
    P.R0 = R0; P.R1 = R1; P.R2 = R2;
    P.wb = wb;
    P.g = g;
    P.inv_I = B->inv_inertia[a];
    P.inv_m = B->inv_mass;
    P.V = B->vel[a];
    P.C = B->center[a];
  }
  if (lane < 4) S.quat[lane] = B->quat[lane];
}

// The step, from the blocks' parts S.sum of the force and torque on the body,
// by the warp that called rigid_prepare. Writes the new state to pose (C, q, V)
// or, with store, to the body.
__device__ __forceinline__ void rigid_finish(BodyDev* B, ClusterShare& S, double* pose, bool store) {
  const int lane = threadIdx.x & 31, a = lane < 3 ? lane : lane % 3;
  constexpr unsigned ALL = 0xffffffffu;
  __syncwarp();
  if (lane < 6) {
    const double t0 = S.sum[0][lane] + S.sum[1][lane], t1 = S.sum[2][lane] + S.sum[3][lane];
    const double t2 = S.sum[4][lane] + S.sum[5][lane], t3 = S.sum[6][lane] + S.sum[7][lane];
    S.total[lane] = (t0 + t1) + (t2 + t3);
  }
  __syncwarp();
  const double* sum = S.total;
  const RigidPrep P = S.prep[a];
  const double V = P.V + sum[a] * P.inv_m;
  const double C = P.C + V;
  const double tb = P.R0 * sum[3] + P.R1 * sum[4] + P.R2 * sum[5];
  const double wb = P.wb + (tb - P.g) * P.inv_I;
  // omega = R wb: row sums across the lanes that hold the columns
  const double p0 = P.R0 * wb, p1 = P.R1 * wb, p2 = P.R2 * wb;
  const double ox = __shfl_sync(ALL, p0, 0) + __shfl_sync(ALL, p0, 1) + __shfl_sync(ALL, p0, 2);
  const double oy = __shfl_sync(ALL, p1, 0) + __shfl_sync(ALL, p1, 1) + __shfl_sync(ALL, p1, 2);
  const double oz = __shfl_sync(ALL, p2, 0) + __shfl_sync(ALL, p2, 1) + __shfl_sync(ALL, p2, 2);
  // lane k < 4: component k of the quaternion
  const double w = S.quat[0], x = S.quat[1], y = S.quat[2], z = S.quat[3];
  const int k = lane & 3;
  const double d = k == 0 ? -ox * x - oy * y - oz * z
                          : (k == 1 ? ox * w + oy * z - oz * y : (k == 2 ? -ox * z + oy * w + oz * x : ox * y - oy * x + oz * w));
  double q = S.quat[k] + 0.5 * d;
  double n2 = q * q;
  n2 += __shfl_xor_sync(ALL, n2, 1);
  n2 += __shfl_xor_sync(ALL, n2, 2);
  // 1/sqrt(n2): two Newton steps from the FP32 value (relative error 1e-7,
  // 1e-14, rounding)
  double rn = (double)rsqrtf((float)n2);
  rn = rn * (1.5 - 0.5 * n2 * rn * rn);
  rn = rn * (1.5 - 0.5 * n2 * rn * rn);
  q *= rn;
  if (lane < 3) {
    if (pose) { pose[a] = C; pose[7 + a] = V; }
    if (store) {
      B->center[a] = C;
      B->vel[a] = V;
      B->omega[a] = a == 0 ? ox : (a == 1 ? oy : oz);
    }
  }
  if (lane < 4) {
    if (pose) pose[3 + k] = q;
    if (store) B->quat[k] = q;
  }
}

// Row a of the rotation matrix of a unit quaternion.
__device__ __forceinline__ void rotation_row(const double* q, int a, double r[3]) {
  const double w = q[0], x = q[1], y = q[2], z = q[3];
  if (a == 0) { r[0] = 1 - 2 * (y * y + z * z); r[1] = 2 * (x * y - w * z); r[2] = 2 * (x * z + w * y); }
  else if (a == 1) { r[0] = 2 * (x * y + w * z); r[1] = 1 - 2 * (x * x + z * z); r[2] = 2 * (y * z - w * x); }
  else { r[0] = 2 * (x * z - w * y); r[1] = 2 * (y * z + w * x); r[2] = 1 - 2 * (x * x + y * y); }
}

// Smallest box around the boxes lo[r], dims[r] of the blocks (dims.w != 0), at
// most CLUSTER_UNION_MAX cells: above that (markers of one body far apart), or
// with no box at all, dims.w = 0.
__device__ __forceinline__ void union_box(const int4* lo, const int4* dims, int4& ulo, int4& udims) {
  int l[3] = {INT_MAX, INT_MAX, INT_MAX}, h[3] = {INT_MIN, INT_MIN, INT_MIN};
#pragma unroll
  for (int r = 0; r < CLUSTER; ++r) {
    const int4 a = lo[r], d = dims[r];
    if (d.w == 0) continue;
    l[0] = min(l[0], a.x); l[1] = min(l[1], a.y); l[2] = min(l[2], a.z);
    h[0] = max(h[0], a.x + d.x); h[1] = max(h[1], a.y + d.y); h[2] = max(h[2], a.z + d.z);
  }
  const long long ex = (long long)h[0] - l[0], ey = (long long)h[1] - l[1], ez = (long long)h[2] - l[2];
  constexpr long long most = CLUSTER_UNION_MAX;
  const bool ok = ex > 0 && ex <= most && ey <= most && ez <= most && ex * ey <= most && ex * ey * ez <= most;
  ulo = make_int4(l[0], l[1], l[2], 0);
  udims = ok ? make_int4((int)ex, (int)ey, (int)ez, 1) : make_int4(0, 0, 0, 0);
}

// Cells of the rows of a body's box that are block `rank`'s (every eighth).
__device__ __forceinline__ int cluster_share(int4 udims, int rank) {
  const int nrows = udims.y * udims.z;
  return nrows > rank ? (nrows - rank + CLUSTER - 1) / CLUSTER * udims.x : 0;
}

// Visits those cells, thread t of n: f(cell index in the lattice, unwrapped x,
// y, z, mask of the blocks whose boxes meet the row). Rows no block's box meets,
// and solid ones, are skipped. The cells are numbered through, so that rows a
// little longer than a warp leave no lanes idle.
template <int GEOM, class F>
__device__ __forceinline__ void cluster_cells(const LatticeDev& L, const int4* lo, const int4* dims, int4 ulo, int4 ud,
                                              int rank, int t, int n, F&& f) {
  const int total = cluster_share(ud, rank);
  const float inv_dx = 1.0f / (float)ud.x, inv_dy = 1.0f / (float)ud.y;
  const int xw0 = wrapi(ulo.x, L.nx);
  for (int c = t; c < total; c += n) {
    int i, ax, iy, iz;
    row_yz(c, ud.x, inv_dx, ax, i);  // c = ax + ud.x i (exact: c < 2^20)
    row_yz(rank + CLUSTER * i, ud.y, inv_dy, iy, iz);
    int y = ulo.y + iy, z = ulo.z + iz;
    unsigned mask = 0u;
#pragma unroll
    for (int q = 0; q < CLUSTER; ++q)
      if (dims[q].w != 0 && (unsigned)(y - lo[q].y) < (unsigned)dims[q].y && (unsigned)(z - lo[q].z) < (unsigned)dims[q].z)
        mask |= 1u << q;
    if (mask == 0u) continue;
    const int uy = y, uz = z;
    if (!fluid_row<GEOM>(L, y, z)) continue;
    f((size_t)L.nx * (y + L.ny * z) + box_x(xw0, ax, L.nx), ulo.x + ax, uy, uz, mask);
  }
}

// A block's views of its membrane: the whole body's positions (integer part
// relative to a common origin, fraction), its part's normals and areas, its
// own vertices' force sums.
struct MembraneArrays {
  const float *sI, *sR;  // [3][nv]
  float *sN, *sA;        // [3][nt_part], [nt_part]
  int* sQ;               // [3][per]
  int nv, nt_part, per, c0, n;
};
struct MembraneModuli {
  float kBT_p, k_b, k_l, k_g, k_v;
};

// Forces on this block's vertices c0 .. c0 + n - 1 of a membrane whose
// positions all blocks of the cluster have written (and synchronised on),
// with S.part_sum and sQ cleared. The sums are left in sQ: fixed point in units of
// `unit`, or floats where unit = 0 (a contribution that is not finite). Returns the thread's largest contribution;
// q_prev: the largest one of the last evaluation. Contains one cluster barrier.
template <int THREADS>
__device__ __forceinline__ float cluster_membrane(ClusterShare& S, const MembraneArrays& W, const MeshPart& P,
                                                  const MeshDev& mesh, const MembraneModuli& Km, float q_prev,
                                                  float& unit) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x;
  const float *sI = W.sI, *sR = W.sR;
  float *sN = W.sN, *sA = W.sA;
  int* sQ = W.sQ;
  float* sF = reinterpret_cast<float*>(sQ);
  const int nv = W.nv, nt_part = W.nt_part, per = W.per, c0 = W.c0, n = W.n;
  const MembraneScale K = membrane_scale(mesh);
  auto dv = [&](int p, int q) {
    return make_float3((sI[p] - sI[q]) + (sR[p] - sR[q]), (sI[nv + p] - sI[nv + q]) + (sR[nv + p] - sR[nv + q]),
                       (sI[2 * nv + p] - sI[2 * nv + q]) + (sR[2 * nv + p] - sR[2 * nv + q]));
  };
  auto normal = [&](int t) { return make_float3(sN[t], sN[nt_part + t], sN[2 * nt_part + t]); };
  // A. normals and areas of the part's triangles; each triangle counts once
  // for the body's area and volume (flag in .w)
  float ap = 0.f, vp = 0.f;
  for (int t = tid; t < P.nt; t += THREADS) {
    const ushort4 Tr = P.tris[t];
    const float3 N = cross(dv(Tr.y, Tr.x), dv(Tr.z, Tr.x));
    const float At = 0.5f * sqrtf(dot(N, N));
    sN[t] = N.x; sN[nt_part + t] = N.y; sN[2 * nt_part + t] = N.z;
    sA[t] = At;
    if (Tr.w) {
      ap += At;
      vp += dot(dv(Tr.x, 0), N) * (1.0f / 6.0f);
    }
  }
  warp_fixed_sum(ap, vp, K, &S.part_sum);
  __syncthreads();
  if (tid < 2 * CLUSTER) {
    const int r = tid >> 1, q = tid & 1;
    cl.map_shared_rank(&S.sum[0][0], r)[6 * rank + q] = S.part_sum.units(q, q == 0 ? K.sa : K.sv);
  }
  // the area and volume terms need the other blocks' sums; the edges do not
  cl.barrier_arrive();
  float qmax = 0.f;
  auto edges = [&](auto&& add) {
    for (int e = tid; e < P.ne; e += THREADS)
      edge_forces(P.edges[e], P.edge_tris[e], P.edge_rest[e], Km.kBT_p, Km.k_b, dv, normal, add);
  };
  const float Sq = q_prev > 0.f ? mesh.qcap / (4.0f * q_prev) : 0.f;
  bool over = !(q_prev > 0.f);
  auto add_fixed = [&](int v, float3 f) {
    const float c = fmaxf(fabsf(f.x), fmaxf(fabsf(f.y), fabsf(f.z)));
    qmax = fmaxf(qmax, c);
    over |= !(c * Sq <= mesh.qcap);
    const int i = v - c0;
    if ((unsigned)i < (unsigned)n) {
      atomicAdd(sQ + i, __float2int_rn(f.x * Sq));
      atomicAdd(sQ + per + i, __float2int_rn(f.y * Sq));
      atomicAdd(sQ + 2 * per + i, __float2int_rn(f.z * Sq));
    }
  };
  const bool scaled = q_prev > 0.f;
  if (scaled) edges(add_fixed);
  cl.barrier_wait();  // partial areas and volumes of all blocks
  double sa = 0.0, sv = 0.0;
#pragma unroll
  for (int r = 0; r < CLUSTER; ++r) {
    sa += S.sum[r][0];
    sv += S.sum[r][1];
  }
  const float cg_ = Km.k_g * ((float)(sa * K.qa - (double)mesh.A0) / mesh.A0);
  const float cv_ = Km.k_v * ((float)(sv * K.qv - (double)mesh.V0) / mesh.V0);
  auto triangles = [&](auto&& add) {
    for (int t = tid; t < P.nt_own; t += THREADS)
      triangle_forces(P.tris[t], normal(t), sA[t], P.area0[t], Km.k_l, cg_, cv_, dv, add);
  };
  if (scaled) triangles(add_fixed);
  const bool redo = __syncthreads_or(over) != 0;
  unit = 1.0f / Sq;
  if (redo) {
    bool is_float;
    auto pass = [&](auto&& add) {
      edges(add);
      triangles(add);
    };
    unit = redo_scatter(pass, sQ, per, n, c0, per, mesh.qcap, qmax, &S.redo_max, is_float);
    __syncthreads();
    if (tid == 0) S.redo_max = 0u;
  }
  return qmax;
}

}  // namespace cluster_detail

// The whole coupling of one body by its cluster (blockDim = CLUSTER_THREADS,
// cluster of CLUSTER blocks along x). KIND: 0 rigid bodies, 1 membranes.
template <int GEOM, int KIND>
__device__ __forceinline__ void cluster_couple(const ClusterArgs& A, ClusterShare& S, unsigned char* smem) {
  using namespace cluster_detail;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const LatticeDev& L = A.L;
  const MarkersDev& m = A.m;
  const size_t M = (size_t)m.M;
  BodyDev* B = A.body;
  const int count = B->count, per = cluster_per(count);
  const int c0 = min(rank * per, count), n = min(per, count - c0), first = B->first + c0;
  const int nv = KIND == 1 ? A.mesh.nv : 0;
  const int nt_part = KIND == 1 ? A.mesh.part_tris : 0;
  int* sCell = reinterpret_cast<int*>(smem);                 // [3][per]
  float* sFrac = reinterpret_cast<float*>(sCell + 3 * per);  // [3][per]
  int* sQ = reinterpret_cast<int*>(sFrac + 3 * per);         // [3][per] membrane sums, then forces
  float* sF = reinterpret_cast<float*>(sQ);
  float* sI = reinterpret_cast<float*>(sQ + 3 * per);        // [3][nv] whole body
  float* sR = sI + 3 * nv;
  float* sN = sR + 3 * nv;                                   // [3][nt_part]
  float* sA = sN + 3 * nt_part;
  int* ibox = reinterpret_cast<int*>(smem) + cluster_fixed_words(count, nv, nt_part);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int a = tid & 3, quad = tid >> 2;
  constexpr int QUADS = CLUSTER_WORKERS / 4, NWORK = CLUSTER_WORKERS / 32;
  const bool worker = warp < NWORK;
  const bool direct = KIND == 0 && B->kind == 3;
  const bool tether = KIND == 0 && !direct;
  // origin of the membrane's integer parts (read before any block moves it)
  int o[3] = {0, 0, 0};
  if (KIND == 1)
    for (int q = 0; q < 3; ++q) o[q] = m.cell[q * M + B->first];
  cl.barrier_arrive();  // the blocks have started, and have read the origin
  if (tid < 3) {
    S.lo_s[tid] = INT_MAX;
    S.hi_s[tid] = INT_MIN;
  }
  if (tid == 0) {
    S.fmax_s = S.redo_max = 0u;
  }
  if (tid < CLUSTER) {
    S.old_lo[tid] = A.boxes[2 * tid];
    S.old_dims[tid] = A.boxes[2 * tid + 1];
  }
  // rigid: lane a < 3 of a quad carries component a of the marker's arm,
  // force and torque
  const int ra = a < 3 ? a : 0, lb = (lane & ~3) + (ra + 1) % 3, lc = (lane & ~3) + (ra + 2) % 3;
  double row[3] = {0, 0, 0}, Ca = 0, kappa = 0, Va = 0, Ob = 0, Oc = 0, acc_f = 0.0, acc_t = 0.0;
  if (KIND == 0 && A.forces) {
    rotation_row(B->quat, ra, row);
    Ca = B->center[ra];
    kappa = B->kappa;
    if (direct) {
      Va = B->vel[ra];
      Ob = B->omega[(ra + 1) % 3];
      Oc = B->omega[(ra + 2) % 3];
    }
  }
  float fm = 0.f;                       // largest force component seen
  int blo = INT_MAX, bhi = INT_MIN;     // bounds of component ra of the cells seen
  __syncthreads();

  // ---- 1. interpolation of step n, advection; rigid forces --------------------
  const bool boxed = S.old_dims[rank].w != 0;
  // (what follows is the markers', bodies' and boxes' own state: the coupling
  // before the finished collision wrote it)
  if (!worker) {
    if (KIND == 0 && A.forces && (direct || rank == 0)) rigid_prepare(B, S);
    await_predecessor();
    dependents_may_launch();
  }
  // The force density and flags that the finished collision read are cleared by
  // the last warp while the others gather (a small body), or by all while the
  // blocks wait for one another.
  int4 old_lo, old_dims;
  union_box(S.old_lo, S.old_dims, old_lo, old_dims);
  const bool clears = A.interp && old_dims.w != 0, ahead = cluster_share(old_dims, 0) <= CLUSTER_CLEAR_AHEAD;
  auto clear_consumed = [&](int t, int n_threads) {
    cluster_cells<GEOM>(L, S.old_lo, S.old_dims, old_lo, old_dims, rank, t, n_threads,
                        [&](size_t gi, int, int, int, unsigned) { L.g[gi] = make_float4(0.f, 0.f, 0.f, 0.f); });
    if (boxed) mark_box_tiles<GEOM>(L, S.old_lo[rank], S.old_dims[rank], t, n_threads, 0);
  };
  if (!worker && clears && ahead) clear_consumed(lane, 32);
  if (worker) {
    // (the next pass's marker is loaded while this one is gathered)
    double Xnext = 0.0, arm_next[3] = {0, 0, 0};
    RawStencil rs_next{};
    auto load_marker = [&](int j) {
      const int k = first + (j < n ? j : 0);
      if (!direct && (A.interp || tether)) Xnext = m.X[(size_t)ra * M + k];
      if (KIND == 0 && A.forces)
#pragma unroll
        for (int q = 0; q < 3; ++q) arm_next[q] = m.ref[q * M + k];
      load_raw(m, k, rs_next);
    };
    if ((warp << 3) < n) load_marker(quad);
    await_predecessor();
    dependents_may_launch();
    for (int j0 = 0; j0 + (warp << 3) < n; j0 += QUADS) {
      const int j = j0 + quad;
      const bool active = j < n, on = active && a < 3;
      const int k = first + (active ? j : 0);
      const size_t off = (size_t)ra * M + k;
      double Xn = Xnext;
      const double arm[3] = {arm_next[0], arm_next[1], arm_next[2]};
      const RawStencil rs = rs_next;
      if (j0 + QUADS + (warp << 3) < n) load_marker(j + QUADS);
      float u = 0.f;  // component ra of the velocity at the marker
      int c = ra == 0 ? rs.c[0] : (ra == 1 ? rs.c[1] : rs.c[2]);
      float fr = ra == 0 ? rs.f[0] : (ra == 1 ? rs.f[1] : rs.f[2]);
      if (A.interp) {
        const int x = wrapi(rs.c[0] - 1 + a, L.nx);
        // all 16 loads of the column first
        float4 v[16];
#pragma unroll
        for (int cz = 0; cz < 4; ++cz)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            int y = rs.c[1] - 1 + b, z = rs.c[2] - 1 + cz;
            const bool fluid = fluid_row<GEOM>(L, y, z);
            const size_t gi = (size_t)L.nx * (y + L.ny * z) + x;
            v[4 * cz + b] = fluid ? L.uw[gi] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (fluid && !boxed && active) L.g[gi] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
        if (!boxed) mark_tiles<GEOM>(L, rs.c[0] - 1, rs.c[1] - 1, rs.c[2] - 1, active, 0);
        const float wxa = axis_weight(rs.f[0], a);
        float wy[4], wz[4];
        axis_weights(rs.f[1], wy);
        axis_weights(rs.f[2], wz);
        float ux = 0.f, uy = 0.f, uz = 0.f;
#pragma unroll
        for (int cz = 0; cz < 4; ++cz)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float wyz = wy[b] * wz[cz];
            ux = fmaf(wyz, v[4 * cz + b].x, ux);
            uy = fmaf(wyz, v[4 * cz + b].y, uy);
            uz = fmaf(wyz, v[4 * cz + b].z, uz);
          }
        ux *= wxa;
        uy *= wxa;
        uz *= wxa;
#pragma unroll
        for (int s = 1; s < 4; s <<= 1) {
          ux += __shfl_xor_sync(0xffffffffu, ux, s);
          uy += __shfl_xor_sync(0xffffffffu, uy, s);
          uz += __shfl_xor_sync(0xffffffffu, uz, s);
        }
        u = ra == 0 ? ux : (ra == 1 ? uy : uz);
        if (active && a == 0) m.U[k] = make_float4(ux, uy, uz, 0.f);
        if (on && !direct) {
          Xn += (double)u;
          split_coord(Xn, c, fr);
          m.X[off] = Xn;
          if (KIND == 0) {
            m.cell[off] = c;
            m.frac[off] = fr;
          }
        }
      } else if (direct && on) {
        const float4 U = m.U[k];
        u = ra == 0 ? U.x : (ra == 1 ? U.y : U.z);
      }
      if (on) {
        sCell[ra * per + j] = c;
        sFrac[ra * per + j] = fr;
        blo = min(blo, c);
        bhi = max(bhi, c);
      }
      if (KIND == 0 && A.forces) {
        const double w = row[0] * arm[0] + row[1] * arm[1] + row[2] * arm[2];
        const double wb = __shfl_sync(0xffffffffu, w, lb), wc = __shfl_sync(0xffffffffu, w, lc);
        // force on the solid
        const double f = direct ? kappa * ((double)u - (Va + Ob * wc - Oc * wb)) : kappa * (Xn - (Ca + w));
        const double fb = __shfl_sync(0xffffffffu, f, lb), fc = __shfl_sync(0xffffffffu, f, lc);
        if (on) {
          const float F = (float)(-f);
          sF[ra * per + j] = F;
          fm = fmaxf(fm, fabsf(F));
          acc_f += f;
          acc_t += wb * fc - wc * fb;
        }
      }
    }
  }
  cl.barrier_wait();  // every block has started and has read the origin
  if (!A.forces) {
    if (clears && !ahead) clear_consumed(tid, CLUSTER_THREADS);
    if (KIND == 1) {
      __syncthreads();
      for (int i = tid; i < 3 * n; i += CLUSTER_THREADS) {
        const int q = i / n, j = i - q * n;
        m.cell[q * M + first + j] = sCell[q * per + j];
        m.frac[q * M + first + j] = sFrac[q * per + j];
      }
    }
    return;  // (nothing remote follows)
  }

  // ---- 2. forces ------------------------------------------------------------
  if constexpr (KIND == 0) {
    if (worker) {
#pragma unroll
      for (int s = 4; s < 32; s <<= 1) {
        acc_f += __shfl_xor_sync(0xffffffffu, acc_f, s);
        acc_t += __shfl_xor_sync(0xffffffffu, acc_t, s);
      }
      if (lane < 3) {
        S.part[warp][lane] = acc_f;
        S.part[warp][3 + lane] = acc_t;
      }
    }
    __syncthreads();
    if (tid < 6 * CLUSTER) {  // this block's sums, to every block
      const int r = tid / 6, q = tid - 6 * r;
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < NWORK; ++w) s += S.part[w][q];
      cl.map_shared_rank(&S.sum[0][0], r)[6 * rank + q] = s;
    }
    for (int j = tid; j < n; j += CLUSTER_THREADS)
      m.F[first + j] = make_float4(sF[j], sF[per + j], sF[2 * per + j], 0.f);
    if (direct) {
      cl.sync();
      if (warp == NWORK) rigid_finish(B, S, S.pose, false);
      __syncthreads();
      rotation_row(S.pose + 3, ra, row);
      Ca = S.pose[ra];
      blo = INT_MAX;
      bhi = INT_MIN;
      for (int j = quad; worker && j < n; j += QUADS) {
        if (a == 3) continue;
        const int k = first + j;
        const double X = Ca + row[0] * m.ref[k] + row[1] * m.ref[M + k] + row[2] * m.ref[2 * M + k];
        int c;
        float f;
        split_coord(X, c, f);
        m.X[ra * M + k] = X;
        m.cell[ra * M + k] = c;
        m.frac[ra * M + k] = f;
        sCell[ra * per + j] = c;
        sFrac[ra * per + j] = f;
        blo = min(blo, c);
        bhi = max(bhi, c);
      }
    }
  } else {
    __syncthreads();
    // own positions to every block of the cluster
    for (int i = tid; i < 3 * n; i += CLUSTER_THREADS) {
      const int q = i / n, j = i - q * n;
      const int ci = sCell[q * per + j];
      const float fc = (float)(ci - o[q]), fr = sFrac[q * per + j];
#pragma unroll
      for (int r = 0; r < CLUSTER; ++r) {
        float* d = cl.map_shared_rank(sI, r);
        d[q * nv + c0 + j] = fc;
        d[3 * nv + q * nv + c0 + j] = fr;
      }
      m.cell[q * M + first + j] = ci;
      m.frac[q * M + first + j] = fr;
    }
    for (int i = tid; i < 3 * per; i += CLUSTER_THREADS) sQ[i] = 0;
    if (tid == 0) S.part_sum = BodySums{};
    if (tid < CLUSTER) S.qmax[tid] = 0u;
    cl.sync();  // positions complete
    const MembraneModuli Km{B->kBT_p, B->k_b, B->k_l, B->k_g, B->k_v};
    float unit;
    float qmax = cluster_membrane<CLUSTER_THREADS>(S, MembraneArrays{sI, sR, sN, sA, sQ, nv, nt_part, per, c0, n},
                                                   mesh_part(A.mesh, rank), A.mesh, Km, B->qmax, unit);
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, s));
    if (lane == 0) atomicMax(cl.map_shared_rank(&S.qmax[0], 0) + rank, __float_as_uint(qmax));
    __syncthreads();
    for (int j = tid; j < n; j += CLUSTER_THREADS) {
      float F[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        F[q] = unit > 0.f ? (float)sQ[q * per + j] * unit : sF[q * per + j];
        sF[q * per + j] = F[q];
        fm = fmaxf(fm, fabsf(F[q]));
      }
      m.F[first + j] = make_float4(F[0], F[1], F[2], 0.f);
    }
  }

  // the body's new state, from all blocks' sums (the last warp of block 0)
  auto update_body = [&]() {
    if constexpr (KIND == 0) {
      rigid_finish(B, S, nullptr, true);
    } else if (lane == 0) {
      float q = 0.f;
#pragma unroll
      for (int r = 0; r < CLUSTER; ++r) q = fmaxf(q, __uint_as_float(S.qmax[r]));
      B->qmax = isfinite(q) ? q : 0.f;
    }
  };
  if (!A.spread) {
    cl.sync();
    if (rank == 0 && !worker) update_body();
    return;  // (block 0 reads its own shared memory only)
  }

  // ---- 3. spreading of step n+1 ----------------------------------------------
  // bounds and largest force of the block's markers
#pragma unroll
  for (int s = 4; s < 32; s <<= 1) {
    blo = min(blo, __shfl_xor_sync(0xffffffffu, blo, s));
    bhi = max(bhi, __shfl_xor_sync(0xffffffffu, bhi, s));
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) fm = fmaxf(fm, __shfl_xor_sync(0xffffffffu, fm, s));
  if (worker && lane < 3) {
    atomicMin(&S.lo_s[lane], blo);
    atomicMax(&S.hi_s[lane], bhi);
  }
  if (lane == 0) atomicMax(&S.fmax_s, __float_as_uint(fm));  // non-negative floats order as their bits
  __syncthreads();
  const long long ex = (long long)S.hi_s[0] - S.lo_s[0] + 4, ey = (long long)S.hi_s[1] - S.lo_s[1] + 4,
                  ez = (long long)S.hi_s[2] - S.lo_s[2] + 4;
  // each extent below cap before the products: no overflow
  const bool own_fits = n > 0 && ex <= A.cap && ey <= A.cap && ez <= A.cap && ex * ey <= A.cap && ex * ey * ez <= A.cap;
  const int4 lo2 = make_int4(S.lo_s[0] - 1, S.lo_s[1] - 1, S.lo_s[2] - 1, 0);
  const int4 dims2 = make_int4(own_fits ? (int)ex : 0, own_fits ? (int)ey : 0, own_fits ? (int)ez : 0, own_fits ? 1 : 0);
  const int vol = dims2.x * dims2.y * dims2.z;
  if (tid < CLUSTER) {
    ClusterShare* R = cl.map_shared_rank(&S, tid);
    R->lo[rank] = lo2;
    R->dims[rank] = dims2;
    R->fmax[rank] = S.fmax_s;
  }
  for (int i = tid; i < (3 * vol + 3) / 4; i += CLUSTER_THREADS)  // (cap is a multiple of 4)
    reinterpret_cast<int4*>(ibox)[i] = make_int4(0, 0, 0, 0);
  LatticeDev Ln = L;
  Ln.g = A.g_next;
  Ln.flags = A.flags_next;
  __syncthreads();
  cl.barrier_arrive();
  if (clears && !ahead) clear_consumed(tid, CLUSTER_THREADS);
  cl.barrier_wait();  // boxes, forces and sums of all blocks
  int4 ulo, udims;
  union_box(S.lo, S.dims, ulo, udims);
  const bool fits = own_fits && udims.w != 0;  // (markers of one body far apart: no box)
  if (tid == 0) {  // (every block has read the old ones)
    A.boxes[2 * rank] = lo2;
    A.boxes[2 * rank + 1] = make_int4(dims2.x, dims2.y, dims2.z, fits ? 1 : 0);
  }
  if (fits) mark_box_tiles<GEOM>(Ln, lo2, dims2);
  unsigned fbits = 0u;
#pragma unroll
  for (int r = 0; r < CLUSTER; ++r) fbits = max(fbits, S.fmax[r]);
  const float fmax = __uint_as_float(fbits);
  const bool any_force = fmax > 0.f;
  // Fixed-point scale as in spread_group, with the bound on a cell's sum taken
  // over the body while spread_group's groups hold a body (the same integers);
  // a larger body, several groups there, takes it over a block's markers, and
  // the sum over the blocks is split below.
  const bool wide = count > XFER_GROUP_MAX;
  const float Sc = any_force ? fminf(33554432.0f, 8589934592.0f / (float)(wide ? per : count)) / fmax : 0.f;
  if (worker) {
    for (int j0 = 0; j0 + (warp << 3) < n; j0 += QUADS) {
      const int j = j0 + quad;
      const bool active = j < n;
      const int jj = active ? j : 0;
      const int bx = sCell[jj] - 1, by = sCell[per + jj] - 1, bz = sCell[2 * per + jj] - 1;
      if (!fits) mark_tiles<GEOM>(Ln, bx, by, bz, active);
      if (!active || !any_force) continue;
      const float wxa = axis_weight(sFrac[jj], a);
      float wy[4], wz[4];
      axis_weights(sFrac[per + jj], wy);
      axis_weights(sFrac[2 * per + jj], wz);
      const float Fx = sF[jj], Fy = sF[per + jj], Fz = sF[2 * per + jj];
      if (fits) {
        const float ax_ = Fx * Sc * wxa, ay_ = Fy * Sc * wxa, az_ = Fz * Sc * wxa;
        int* p0 = ibox + (bx - lo2.x + a) + dims2.x * ((by - lo2.y) + dims2.y * (bz - lo2.z));
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float wyz = wy[b] * wz[c];
            int* p = p0 + dims2.x * (b + dims2.y * c);
            atomicAdd(p, fixed_mul(ax_, wyz));
            atomicAdd(p + vol, fixed_mul(ay_, wyz));
            atomicAdd(p + 2 * vol, fixed_mul(az_, wyz));
          }
      } else {
        const int x = wrapi(bx + a, L.nx);
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            int y = by + b, z = bz + c;
            if (!fluid_row<GEOM>(L, y, z)) continue;
            const float w = wxa * (wy[b] * wz[c]);
            atomicAdd(Ln.g + (size_t)L.nx * (y + L.ny * z) + x, make_float4(Fx * w, Fy * w, Fz * w, 0.f));
          }
      }
    }
    cl.barrier_arrive();
  } else {
    cl.barrier_arrive();
    if (rank == 0) update_body();
  }
  cl.barrier_wait();  // the boxes are complete
  if (any_force && udims.w != 0) {
    const float inv = 1.0f / Sc;
    cluster_cells<GEOM>(L, S.lo, S.dims, ulo, udims, rank, tid, CLUSTER_THREADS, [&](size_t gi, int ux, int uy, int uz, unsigned mask) {
      int q[3] = {0, 0, 0}, lo4[3] = {0, 0, 0};
#pragma unroll
      for (int r = 0; r < CLUSTER; ++r) {
        const int4 lo = S.lo[r], d = S.dims[r];
        const int ox = ux - lo.x, v = d.x * d.y * d.z;
        int t[3] = {0, 0, 0};
        if (((mask >> r) & 1u) != 0u && (unsigned)ox < (unsigned)d.x) {
          const int* p = cl.map_shared_rank(ibox, r) + (ox + d.x * ((uy - lo.y) + d.y * (uz - lo.z)));
          t[0] = p[0];
          t[1] = p[v];
          t[2] = p[2 * v];
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          if (wide) {  // eight sums below 2^30: their high parts and low 4 bits apart
            q[i] += t[i] >> 4;
            lo4[i] += t[i] & 15;
          } else {
            q[i] += t[i];
          }
        }
      }
      if ((q[0] | q[1] | q[2] | lo4[0] | lo4[1] | lo4[2]) == 0) return;
      float g[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) g[i] = (wide ? fmaf((float)q[i], 16.0f, (float)lo4[i]) : (float)q[i]) * inv;
      atomicAdd(Ln.g + gi, make_float4(g[0], g[1], g[2], 0.f));
    });
  }
  cl.sync();  // no block leaves while another reads its shared memory
}

}  // namespace ibm
