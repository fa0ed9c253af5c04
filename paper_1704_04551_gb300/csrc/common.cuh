// Device-side definitions shared by the kernels of the coupled IBM-LBM step.
// Lattice: D3Q19 (Sec. 2.1 of arXiv:1704.04551), c_s^2 = 1/3 (Eq. viscosity).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ibm {

constexpr int Q = 19;

// Thread blocks that share one body's coupling where there are few bodies
// (cluster_body.cuh; the portable cluster size).
constexpr int CLUSTER = 8;

// Velocities in the public D3Q19 order: rest, +-x, +-y, +-z, then the face
// diagonals in opposite pairs, so that opposite(i) = i + 1 for odd i and
// i - 1 for even i > 0.
__host__ __device__ constexpr int cx(int i) {
  constexpr int v[Q] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
  return v[i];
}
__host__ __device__ constexpr int cy(int i) {
  constexpr int v[Q] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
  return v[i];
}
__host__ __device__ constexpr int cz(int i) {
  constexpr int v[Q] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
  return v[i];
}
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
__host__ __device__ constexpr float wgt(int i) {
  return i == 0 ? (1.0f / 3.0f) : (i < 7 ? (1.0f / 18.0f) : (1.0f / 36.0f));
}
__host__ __device__ constexpr double wgt_d(int i) {
  return i == 0 ? (1.0 / 3.0) : (i < 7 ? (1.0 / 18.0) : (1.0 / 36.0));
}
// Power-of-two scale of the half-precision deviation store, ~1/w_i.
__host__ __device__ constexpr float dev_scale(int i) { return i == 0 ? 4.0f : (i < 7 ? 16.0f : 32.0f); }

enum Geometry : int { GEOM_PERIODIC = 0, GEOM_YWALLS = 1, GEOM_TUBE = 2 };
enum Storage : int { STORE_F32 = 0, STORE_F16 = 1, STORE_BF16 = 2 };

// Tiles used to mark where markers touch the lattice: 32 (x) x 4 x 4 cells.
constexpr int TILE_X_SHIFT = 5, TILE_Y_SHIFT = 2, TILE_Z_SHIFT = 2;

// Programmatic dependent launch: a kernel launched by launch_after(..., true)
// may start while its predecessor in the stream still runs, once all the
// predecessor's blocks have called dependents_may_launch (or ended). Before
// await_predecessor returns it may read only what was complete before the
// predecessor started. The collision and the coupling kernels of a step
// await theirs before they let their successor go, so a kernel may read,
// ahead of the wait, whatever the kernel before its predecessor wrote: the
// coupling its markers. (In an ordinary launch both calls are no-ops.)
__device__ __forceinline__ void await_predecessor() { cudaGridDependencySynchronize(); }
__device__ __forceinline__ void dependents_may_launch() { cudaTriggerProgrammaticLaunchCompletion(); }

template <class... P, class... A>
inline void launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool programmatic,
                         A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = programmatic ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Exact n / d for 32-bit n (Granlund & Montgomery, "Division by invariant
// integers using multiplication", 1994): four instructions.
struct FastDiv {
  unsigned m, s1, s2;
};
inline FastDiv fast_div(unsigned d) {
  int l = 0;
  while ((1ull << l) < d) ++l;
  const unsigned m = (unsigned)(((1ull << 32) * ((1ull << l) - d)) / d + 1);
  return {m, l < 1 ? (unsigned)l : 1u, l < 1 ? 0u : (unsigned)l - 1u};
}
__device__ __forceinline__ unsigned divide(unsigned n, const FastDiv& d) {
  const unsigned t = __umulhi(d.m, n);
  return (t + ((n - t) >> d.s1)) >> d.s2;
}

struct LatticeDev {
  int nx, ny, nz;
  int N;                 // nx*ny*nz (< 2^31)
  int geometry;
  float omega;           // 1/tau
  float guo_pre;         // 1 - 1/(2 tau)
  float wall_u0, wall_u1;
  float yc, zc, R2;      // tube axis and squared radius
  float g0x, g0y, g0z;   // uniform body force density
  int ntx, nty, ntz;     // tile grid
  void* pop;             // [19][N] in the storage type
  float4* uw;            // moments of the last collision: (ux, uy, uz, rho - 1) [N]
  // Force density and touched-tile flags: the step's spreading adds into g
  // (zero at that point) and marks flags, the collision reads g where flags
  // is set, and the interpolation, which sweeps the same boxes of cells
  // afterwards, writes g back to zero there (in its latency-bound box load,
  // not in the bandwidth-bound collision). flags is cleared at the start of
  // each step (couplings by clusters have two of each: a coupling clears what
  // its collision read and sets the other).
  float4* g;             // spread force density (gx, gy, gz, 0) [N]
  uint8_t* flags;        // [ntx*nty*ntz]: tile touched by a marker stencil this step
  int* status;           // device status word (0 = OK)
  FastDiv by_nx;         // cell of the fluid rows -> (row, x)
};

// One lattice row (fixed y, z; all x) that holds fluid. Solidity depends on
// (y, z) only in every geometry, so a row is all fluid or all solid and the
// collide kernel runs over the fluid rows alone.
struct RowInfo {
  int base;              // idx of (0, y, z)
  int smask;             // bit (dy+1)*3 + (dz+1): the row at (y+dy, z+dz) is solid
  int oyp, oym, ozp, ozm;// wrapped element offsets to the y+-1, z+-1 rows
  int y;
  int trow;              // tile-row offset ntx * ((y >> 2) + nty * (z >> 2))
};

// A contiguous run of markers handled by one thread block in the transfer
// kernels (a body, or part of one, or a run of passive tracers).
struct MarkerGroup {
  int first, count;
  int flags;  // GROUP_FIXED: positions set by a rigid body, not advected
};
constexpr int GROUP_FIXED = 1;

// Solid test of a node with wrapped x and (for walls/tube) raw y, z.
__device__ __forceinline__ bool solid_yz(const LatticeDev& L, int y, int z) {
  if (L.geometry == GEOM_YWALLS) return (unsigned)y >= (unsigned)L.ny;
  if (L.geometry == GEOM_TUBE) {
    if ((unsigned)y >= (unsigned)L.ny || (unsigned)z >= (unsigned)L.nz) return true;
    float dy = (float)y - L.yc, dz = (float)z - L.zc;
    return dy * dy + dz * dz > L.R2;
  }
  return false;
}

__device__ __forceinline__ int wrapi(int v, int n) {
  v = v % n;
  return v < 0 ? v + n : v;
}

// Two FP32 operations in one instruction (Blackwell's packed FP32 pipe): each
// half rounds as the scalar operation does.
struct F32x2 {
  unsigned long long v;
};
__device__ __forceinline__ F32x2 pack2(float a, float b) {
  F32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(F32x2 p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
}
__device__ __forceinline__ F32x2 fma2(F32x2 a, F32x2 b, F32x2 c) {
  F32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F32x2 mul2(F32x2 a, F32x2 b) {
  F32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F32x2 add2(F32x2 a, F32x2 b) {
  F32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F32x2 both(float a) { return pack2(a, a); }
__device__ __forceinline__ F32x2 sub2(F32x2 a, F32x2 b) { return fma2(b, both(-1.0f), a); }

// ---- population storage ---------------------------------------------------
template <int S> struct Store;
template <> struct Store<STORE_F32> {
  using T = float;
  template <int I> __device__ static __forceinline__ float ld(const T* p) { return *p; }
  template <int I> __device__ static __forceinline__ void st(T* p, float v) { *p = v; }
};
template <> struct Store<STORE_F16> {
  using T = __half;
  template <int I> __device__ static __forceinline__ float ld(const T* p) {
    return __half2float(*p) * (1.0f / dev_scale(I));
  }
  template <int I> __device__ static __forceinline__ void st(T* p, float v) {
    *p = __float2half_rn(v * dev_scale(I));
  }
};
template <> struct Store<STORE_BF16> {
  using T = __nv_bfloat16;
  template <int I> __device__ static __forceinline__ float ld(const T* p) {
    return __bfloat162float(*p) * (1.0f / dev_scale(I));
  }
  template <int I> __device__ static __forceinline__ void st(T* p, float v) {
    *p = __float2bfloat16_rn(v * dev_scale(I));
  }
};

// ---- markers and bodies ---------------------------------------------------
struct BodyDev {
  int kind;              // 0 membrane, 1 rigid
  int first, count;
  float kBT_p, k_b, k_l, k_g, k_v;
  double kappa, mass, inertia[3];
  double inv_mass, inv_inertia[3];
  double center[3], quat[4], vel[3], omega[3];
  float qmax;  // membranes: largest force contribution component of the last step (0: none yet)
  float l0;    // filaments: rest bond length
};

struct MeshDev {
  int nv, nt, ne;
  // Template topology packed in one buffer of 16-byte-aligned sections:
  // edges ushort4 (a, b, c, d): edge a->b, wing c in the triangle with a->b,
  // d in the other; edge_tris ushort2 (t1, t2): those two triangles;
  // edge_rest float4 (l0, cos theta0, sin theta0, -); tris ushort4 (v0, v1, v2, -); area0 float;
  // per-vertex CSR lists ve_start/ve of (edge << 2 | role a,b,c,d) and
  // vt_start/vt of (triangle << 2 | slot), all unsigned short.
  const unsigned char* packed;
  int packed_bytes;  // multiple of 16
  int off_edges, off_edge_tris, off_edge_rest, off_tris, off_area0, off_ve_start, off_ve, off_vt_start, off_vt;
  // The template in CLUSTER parts of consecutive vertices (cluster_body.cuh):
  // a table [CLUSTER][8] of (edges, triangles, triangles that touch the part,
  // offsets of edges, edge_tris, edge_rest, tris, area0), each part with its
  // own copy of the edges that touch its vertices and of their triangles.
  int off_parts, part_tris;  // part_tris: largest triangle count of a part
  int work_floats;   // per-body shared work area: 9 nv + 4 nt words
  float A0, V0;
  float fix_a, fix_v;  // powers of two: fixed-point scales of the area and volume sums
  float qcap;        // fixed-point force scatter: largest |contribution| in units, such
                     // that a vertex's sum of all its contributions fits in int32
};

struct MarkersDev {
  int M;
  double* X;          // [3][M] positions (FP64, unwrapped)
  float4* U;          // (Ux, Uy, Uz, 0) [M]
  float4* F;          // (Fx, Fy, Fz, 0) [M]
  const double* ref;  // rigid body-frame offsets [3][M]
  // Stencil cache of the current positions: cell[a][k] = floor(X_a,k) and
  // frac[a][k] = X_a,k - floor(X_a,k) rounded once to FP32. Written when the
  // positions change (set_markers, advection) so that the force, spreading
  // and interpolation kernels need no FP64 arithmetic.
  int* cell;          // [3][M]
  float* frac;        // [3][M]
};

// X = c + f with c = floor(X) and f = X - c rounded once to FP32, for
// |X| < 2^30. Integer arithmetic on the bits of X: an SM does 2 FP64 lanes a
// cycle here, and floor, conversion, subtraction and conversion in FP64 cost
// four of them per coordinate (of the fused kernel's 49 us per body about 2).
// The result is the same, bit for bit.
__device__ __forceinline__ void split_coord(double X, int& c, float& f) {
  const unsigned hw = (unsigned)__double2hiint(X);
  const int e = (int)((hw >> 20) & 0x7ffu) - 1023;
  if (e < -8 || e > 30) {  // tiny (or out of range): the plain way
    const double fl = floor(X);
    c = (int)fl;
    f = (float)(X - fl);
    return;
  }
  const unsigned long long mant =
      ((unsigned long long)((hw & 0xfffffu) | 0x100000u) << 32) | (unsigned)__double2loint(X);
  const long long v = (int)hw < 0 ? -(long long)mant : (long long)mant;  // X 2^(52 - e)
  const int s = 52 - e;                                                   // 22 .. 60
  c = (int)(v >> s);
  const unsigned long long q = (unsigned long long)v << (64 - s);  // fraction, 2^-64 units
  // one rounding: normalised to 32 significant bits, with a sticky bit for
  // the rest (an FP32 significand has 24)
  const int z = min(__clzll((long long)q), 64 - 32);
  const unsigned long long t = q << z;
  const unsigned h = (unsigned)(t >> 32) | ((unsigned)t != 0u ? 1u : 0u);
  f = __uint2float_rn(h) * __int_as_float((127 - 32 - z) << 23);
}

// Stencil cache of one marker coordinate: floor and fractional part.
__device__ __forceinline__ void cache_coord(const MarkersDev& m, size_t off, double X) {
  int c;
  float f;
  split_coord(X, c, f);
  m.cell[off] = c;
  m.frac[off] = f;
}

}  // namespace ibm
