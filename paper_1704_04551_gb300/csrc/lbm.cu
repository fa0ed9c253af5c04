// Lattice-Boltzmann kernels: fused BGK collision + Guo forcing + streaming on
// a single in-place population array (AA access pattern), and the kernels
// that initialise, import, export and check that array.
//
// Method: Sec. 2.1 of arXiv:1704.04551 — Eq. lbm (stream + BGK collide +
// force term), Eq. BGKequilibrium (equilibrium), Eq. rho_u (moments with the
// half-force shift), the Guo term F_i, Eq. viscosity (tau).
//
// AA pattern (one array, each cell reads and writes the same 19 slots):
//   even step: f_i(x) is read from A[x][i]; the post-collision f*_i(x) is
//              written to A[x][opp(i)] (a bounced value carries the
//              moving-wall term already);
//   odd step:  f_i(x) is read from A[x - c_i][opp(i)] (from A[x][i] when
//              x - c_i is solid); f*_i(x) is written to A[x + c_i][i], or,
//              when x + c_i is solid, bounced to A[x][opp(i)].
// After an odd step the array holds f(t+1) in the natural layout.
// Populations are stored as deviations d_i = f_i - w_i (scaled in FP16/BF16)
// and all arithmetic is FP32 in deviation form, which keeps the O(u)
// information of f_i ~ w_i in the significand.
#include "common.cuh"
#include "internal.h"
#include "lbm_cell.cuh"

namespace ibm {


// Fused collide-stream-force kernel: one thread per fluid cell, the cells of
// the fluid rows numbered through (row, x), so that the warps of a lattice
// whose rows are no multiple of 32 or 128 cells long stay full and read whole
// lines. Row data (offsets of the neighbouring rows, which of them are solid)
// come from the precomputed row table.
constexpr int COLLIDE_THREADS = 128;
// Resident blocks per SM the register budget is sized for (more blocks,
// more loads in flight; fewer registers): measured best at 256^3 with 10
// (48 registers) for the local even step, 9 (56 registers) for the
// neighbour-addressed odd step in FP32 and 10 for it in the half-precision
// formats. FP32: even 324 -> 316 us, odd 356 -> 331 us against 8 blocks (64
// registers); FP16 even 244 -> 228 us.
template <int S, int ODD>
constexpr int collide_min_blocks() {
  return (S == STORE_F32 && ODD) ? 9 : 10;
}

// CHAINED: launched ahead of the end of the coupling before it (lattices of at
// most CHAINED_CELLS_MAX cells). A variant of its own: the test of an argument
// cost the large launches 1-5 %, and the wait after the populations' loads,
// which the coupling leaves alone, 6 % (FP16 at 256^3: 186 -> 198 us).
template <int S, int ODD, int GEOM, bool DENSE, bool IDX32, bool CHAINED>
__global__ void __launch_bounds__(COLLIDE_THREADS, (collide_min_blocks<S, ODD>())) k_collide(LatticeDev L, const RowInfo* __restrict__ rows,
                                                                unsigned n_cells) {
  const unsigned t = blockIdx.x * (unsigned)COLLIDE_THREADS + threadIdx.x;
  if (t >= n_cells) return;
  const unsigned r = divide(t, L.by_nx);
  const int x = (int)(t - r * (unsigned)L.nx);
  const RowInfo R = rows[r];
  if constexpr (CHAINED) {
    await_predecessor();
    dependents_may_launch();
  }
  // In the neighbour-addressed (odd) step, rows without solid neighbours
  // (all but a ring of rows along walls) skip the bounce-back tests; few warps
  // lie in two rows of different kinds. (The even step reads and
  // writes its own cell only: a second copy there only cost registers.)
  if constexpr (ODD == 1 && GEOM != GEOM_PERIODIC) {
    if (R.smask == 0) {
      collide_cell<S, ODD, GEOM, DENSE, IDX32, true>(L, R, x);
      return;
    }
  }
  collide_cell<S, ODD, GEOM, DENSE, IDX32>(L, R, x);
}

// Half-precision storage on lattices with even rows: two cells per thread
// (collide_pair); in the odd step rows with solid neighbours cell by cell.
// 256^3 tube, FP16: even step 186 -> 158 us, odd 208 -> 187 us; 7 resident
// blocks (72 registers) measured best (even: 6: 166, 8: 160 us). From
// PAIR_CELLS_MIN fluid cells on: below, the single-cell kernel is one wave, and
// half the threads only wait longer (60x47x33, odd: 9.0 against 10.6 us). Mean
// of both steps, pairs / single, cubes of 32, 48, 60, 64, 80, 96, 128: periodic
// 6.3/6.3, 6.9/7.2, 8.3/8.5, 8.3/9.3, 11.4/13.4, 15.5/18.6, 30.0/38.0; y walls
// 7.3/6.3, 7.7/7.5, 9.4/9.4, 8.8/10.0, 12.5/13.9, 16.7/19.6, 30.6/39.1 us.
constexpr unsigned PAIR_CELLS_MIN = 1u << 18;
constexpr int PAIR_MIN_BLOCKS = 7;
template <int S, int ODD, int GEOM, bool DENSE, bool IDX32>
__global__ void __launch_bounds__(COLLIDE_THREADS, PAIR_MIN_BLOCKS) k_collide_pair(LatticeDev L, const RowInfo* __restrict__ rows,
                                                                      unsigned n_cells) {
  const unsigned t = 2u * (blockIdx.x * (unsigned)COLLIDE_THREADS + threadIdx.x);
  if (t >= n_cells) return;
  const unsigned r = divide(t, L.by_nx);
  const int x = (int)(t - r * (unsigned)L.nx);
  const RowInfo R = rows[r];
  if constexpr (ODD == 1 && GEOM != GEOM_PERIODIC) {
    if (R.smask != 0) {
#pragma unroll 1
      for (int q = 0; q < 2; ++q) collide_cell<S, ODD, GEOM, DENSE, IDX32>(L, R, x + q);
      return;
    }
  }
  collide_pair<S, ODD, GEOM, DENSE, IDX32>(L, R, x);
}

// Equilibrium initialisation from the moments in uw (ux, uy, uz, rho - 1).
template <int S, int GEOM>
__global__ void k_init_equilibrium(LatticeDev L) {
  using P = Pop<S>;
  using T = typename P::T;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= L.N) return;
  Cell c;
  T* A = reinterpret_cast<T*>(L.pop);
  const size_t N = (size_t)L.N;
  if (!make_cell<GEOM>(L, idx, c)) {
#pragma unroll
    for (int i = 0; i < Q; ++i) P::st(A + i * N + idx, i, 0.f);
    L.uw[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const float4 m = L.uw[idx];
  const float rho = 1.0f + m.w;
  const float usq15 = 1.5f * (m.x * m.x + m.y * m.y + m.z * m.z);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float cu = cx(i) * m.x + cy(i) * m.y + cz(i) * m.z;
    P::st(A + i * N + idx, i, wgt(i) * (m.w + rho * (3.0f * cu + 4.5f * cu * cu - usq15)));
  }
}

// Natural-layout populations f_i = w_i + d_i, FP64 [19][N]; ODD_NEXT = the
// array is in the post-even-step layout.
template <int S, int GEOM, bool ODD_NEXT>
__global__ void k_export(LatticeDev L, double* out) {
  using P = Pop<S>;
  using T = typename P::T;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= L.N) return;
  const T* A = reinterpret_cast<const T*>(L.pop);
  const size_t N = (size_t)L.N;
  Cell c;
  if (!make_cell<GEOM>(L, idx, c)) {
    for (int i = 0; i < Q; ++i) out[i * N + idx] = 0.0;
    return;
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    float d;
    if (!ODD_NEXT || i == 0) {
      d = P::ld(A + i * N + idx, i);
    } else {
      const bool sol = (GEOM != GEOM_PERIODIC) && nb_solid(c, i, -1);
      d = sol ? P::ld(A + i * N + idx, i) : P::ld(A + opp(i) * N + (idx + nb_off(c, i, -1)), opp(i));
    }
    out[i * N + idx] = wgt_d(i) + (double)d;
  }
}

template <int S>
__global__ void k_import(LatticeDev L, const double* in) {
  using P = Pop<S>;
  using T = typename P::T;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= L.N) return;
  T* A = reinterpret_cast<T*>(L.pop);
  const size_t N = (size_t)L.N;
#pragma unroll
  for (int i = 0; i < Q; ++i) P::st(A + i * N + idx, i, (float)(in[i * N + idx] - wgt_d(i)));
}

// Moments between the API's FP64 layout (rho [N], u [3][N]) and the
// lattice's (u, rho - 1) float4 array: set_lattice's input before the
// equilibrium initialisation, get_fields' output (solid cells report 0).
__global__ void k_set_moments(LatticeDev L, const double* rho, const double* u) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.N) return;
  const size_t N = (size_t)L.N;
  const double r = rho ? rho[i] : 1.0;
  L.uw[i] = make_float4(u ? (float)u[i] : 0.f, u ? (float)u[N + i] : 0.f, u ? (float)u[2 * N + i] : 0.f,
                        (float)(r - 1.0));
}

__global__ void k_get_moments(LatticeDev L, double* rho, double* u) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.N) return;
  const size_t N = (size_t)L.N;
  const int t = i / L.nx;
  const bool fl = !solid_yz(L, t % L.ny, t / L.ny);
  const float4 v = L.uw[i];
  if (rho) rho[i] = fl ? 1.0 + (double)v.w : 0.0;
  if (u) {
    u[i] = fl ? (double)v.x : 0.0;
    u[N + i] = fl ? (double)v.y : 0.0;
    u[2 * N + i] = fl ? (double)v.z : 0.0;
  }
}

// Sum of floats as three unevaluated parts: hi is the rounded sum, mid collects
// the exact errors of its additions (Knuth's two-sum), lo those of mid's.
struct FloatSum {
  float hi = 0.f, mid = 0.f, lo = 0.f;
  static __device__ __forceinline__ float two_sum(float& a, float x) {  // a += x, returns the error
    const float s = __fadd_rn(a, x), b = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, b)), __fsub_rn(x, b));
    a = s;
    return e;
  }
  __device__ __forceinline__ void add_mid(float x) { lo = __fadd_rn(lo, two_sum(mid, x)); }
  __device__ __forceinline__ void add(float x) { add_mid(two_sum(hi, x)); }
  __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
};

// Sums of the last collision's moments over fluid cells, max |u|, and the
// finiteness check. out: [0] sum(rho - 1), [1..3] sum rho u, [4] number of
// fluid cells; *umax2_bits: max |u|^2 as float bits (atomicMax on the bits
// orders non-negative floats).
//
// An SM does 2 FP64 lanes a cycle here, and a cell's conversions, products and
// sums took 11 of them: 2.56 ms at 512^3, where reading the moments takes 0.32.
// So a thread sums up to 16 cells in three floats each (rho u as u + w u, the
// product with its exact error), whose rounding lies below FP64's, and adds
// them to its FP64 sums: 1.5 (3 with 8 cells) FP64 operations a cell. One step
// with its sums: 131x96x110 117 -> 87 us, 211x163x149 288 -> 205 (a few us of
// it the collide's). Largest error of the momentum over four sizes: 1.15e-17 ->
// 3.5e-18 of the sum of magnitudes (with two floats 6e-17). Values past 1e15,
// where a float sum could overflow, and non-finite ones are added in FP64.
// Eight independent loads per thread; lattices that would not fill the chip
// with 16 cells a thread take 8.
constexpr float DIAG_LIMIT = 1e15f;
constexpr int DIAG_LOADS = 8;
__global__ void __launch_bounds__(256) k_diagnostics(LatticeDev L, const RowInfo* __restrict__ rows, unsigned n,
                                                     int rounds, double* out, unsigned* umax2_bits) {
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  float m2 = 0.f;
  bool bad = false;
  const unsigned span = (unsigned)rounds * DIAG_LOADS * 256;
  for (unsigned base = blockIdx.x * span; base < n; base += gridDim.x * span) {
    FloatSum p0, p1, p2, p3;
    for (int round = 0; round < rounds; ++round) {
      const unsigned first = base + (unsigned)round * (DIAG_LOADS * 256) + threadIdx.x;
      float4 v[DIAG_LOADS];
#pragma unroll
      for (int j = 0; j < DIAG_LOADS; ++j) {
        const unsigned t = first + j * 256;
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t < n) {
          const unsigned r = divide(t, L.by_nx);
          v[j] = L.uw[rows[r].base + (int)(t - r * (unsigned)L.nx)];
        }
      }
#pragma unroll
      for (int j = 0; j < DIAG_LOADS; ++j) {
        const float4 m = v[j];
        const float q = m.x * m.x + m.y * m.y + m.z * m.z;
        m2 = fmaxf(m2, q);
        if (q < DIAG_LIMIT * DIAG_LIMIT && fabsf(m.w) < DIAG_LIMIT) {  // (false for NaN)
          auto add = [&](FloatSum& p, float u) {
            const float wu = __fmul_rn(m.w, u);
            p.add(u);
            p.add(wu);
            p.add_mid(__fmaf_rn(m.w, u, -wu));
          };
          p0.add(m.w);
          add(p1, m.x);
          add(p2, m.y);
          add(p3, m.z);
        } else {
          const double rho = 1.0 + (double)m.w;
          s0 += (double)m.w;
          s1 += rho * m.x; s2 += rho * m.y; s3 += rho * m.z;
          bad = bad || !(isfinite(m.x) && isfinite(m.y) && isfinite(m.z) && isfinite(m.w));
        }
      }
    }
    s0 += p0.value();
    s1 += p1.value();
    s2 += p2.value();
    s3 += p3.value();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    s3 += __shfl_xor_sync(0xffffffffu, s3, o);
    m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, o));
  }
  bad = __any_sync(0xffffffffu, bad);
  __shared__ double sh[8][4];
  __shared__ float shm[8];
  __shared__ int shbad;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) shbad = 0;
  __syncthreads();
  if (lane == 0) {
    sh[warp][0] = s0; sh[warp][1] = s1; sh[warp][2] = s2; sh[warp][3] = s3;
    shm[warp] = m2;
    if (bad) shbad = 1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    float mm = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a0 += sh[w][0]; a1 += sh[w][1]; a2 += sh[w][2]; a3 += sh[w][3];
      mm = fmaxf(mm, shm[w]);
    }
    atomicAdd(out + 0, a0);
    atomicAdd(out + 1, a1);
    atomicAdd(out + 2, a2);
    atomicAdd(out + 3, a3);
    if (blockIdx.x == 0) atomicAdd(out + 4, (double)n);
    if (shbad) {
      atomicExch(L.status, 1);
      atomicMax(umax2_bits, 0x7f800000u);  // +inf
    } else {
      atomicMax(umax2_bits, __float_as_uint(mm));
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
namespace {
inline unsigned blocks_for(int n) { return (unsigned)((n + 255) / 256); }

template <int S, int GEOM>
void launch_collide_g(const LatticeDev& L, const RowInfo* rows, int n_rows, bool odd, bool dense, bool early, cudaStream_t st) {
  const unsigned n_cells = (unsigned)n_rows * (unsigned)L.nx;  // <= N < 2^31
  const unsigned block = COLLIDE_THREADS, grid = (n_cells + block - 1) / block;
  // 32-bit element offsets in the odd step while 19 N < 2^32 (a build with
  // IBM_FORCE_IDX64 defined always takes the 64-bit variant, so that the
  // parity tests reach it on small lattices)
#ifdef IBM_FORCE_IDX64
  const bool idx32 = false;
#else
  const bool idx32 = (unsigned long long)Q * (unsigned long long)L.N < (1ull << 32);
#endif
  auto launch = [&](auto kernel) { launch_after(kernel, grid, block, 0, st, early, L, rows, n_cells); };
  if (early) {  // (a small lattice: 32-bit offsets)
    if (odd && dense) launch(k_collide<S, 1, GEOM, true, true, true>);
    else if (odd) launch(k_collide<S, 1, GEOM, false, true, true>);
    else if (dense) launch(k_collide<S, 0, GEOM, true, false, true>);
    else launch(k_collide<S, 0, GEOM, false, false, true>);
    return;
  }
  if constexpr (S != STORE_F32) {
    if (L.nx % 2 == 0 && n_cells >= PAIR_CELLS_MIN) {
      const unsigned pairs = (n_cells / 2 + block - 1) / block;
      auto launch2 = [&](auto kernel) { launch_after(kernel, pairs, block, 0, st, false, L, rows, n_cells); };
      if (odd && idx32) {
        if (dense) launch2(k_collide_pair<S, 1, GEOM, true, true>);
        else launch2(k_collide_pair<S, 1, GEOM, false, true>);
      } else if (odd) {
        if (dense) launch2(k_collide_pair<S, 1, GEOM, true, false>);
        else launch2(k_collide_pair<S, 1, GEOM, false, false>);
      } else {
        if (dense) launch2(k_collide_pair<S, 0, GEOM, true, false>);
        else launch2(k_collide_pair<S, 0, GEOM, false, false>);
      }
      return;
    }
  }
  if (odd && idx32) {
    if (dense) launch(k_collide<S, 1, GEOM, true, true, false>);
    else launch(k_collide<S, 1, GEOM, false, true, false>);
  } else if (odd) {
    if (dense) launch(k_collide<S, 1, GEOM, true, false, false>);
    else launch(k_collide<S, 1, GEOM, false, false, false>);
  } else {
    if (dense) launch(k_collide<S, 0, GEOM, true, false, false>);
    else launch(k_collide<S, 0, GEOM, false, false, false>);
  }
}
template <int S>
void launch_collide_s(const LatticeDev& L, const RowInfo* rows, int n_rows, bool odd, bool dense, bool early, cudaStream_t st) {
  switch (L.geometry) {
    case GEOM_PERIODIC: launch_collide_g<S, GEOM_PERIODIC>(L, rows, n_rows, odd, dense, early, st); break;
    case GEOM_YWALLS: launch_collide_g<S, GEOM_YWALLS>(L, rows, n_rows, odd, dense, early, st); break;
    default: launch_collide_g<S, GEOM_TUBE>(L, rows, n_rows, odd, dense, early, st); break;
  }
}
template <int S, int GEOM>
void launch_init_g(const LatticeDev& L, cudaStream_t st) {
  k_init_equilibrium<S, GEOM><<<blocks_for(L.N), 256, 0, st>>>(L);
}
template <int S>
void launch_init_s(const LatticeDev& L, cudaStream_t st) {
  switch (L.geometry) {
    case GEOM_PERIODIC: launch_init_g<S, GEOM_PERIODIC>(L, st); break;
    case GEOM_YWALLS: launch_init_g<S, GEOM_YWALLS>(L, st); break;
    default: launch_init_g<S, GEOM_TUBE>(L, st); break;
  }
}
template <int S, int GEOM>
void launch_export_g(const LatticeDev& L, bool odd_next, double* out, cudaStream_t st) {
  if (odd_next) k_export<S, GEOM, true><<<blocks_for(L.N), 256, 0, st>>>(L, out);
  else k_export<S, GEOM, false><<<blocks_for(L.N), 256, 0, st>>>(L, out);
}
template <int S>
void launch_export_s(const LatticeDev& L, bool odd_next, double* out, cudaStream_t st) {
  switch (L.geometry) {
    case GEOM_PERIODIC: launch_export_g<S, GEOM_PERIODIC>(L, odd_next, out, st); break;
    case GEOM_YWALLS: launch_export_g<S, GEOM_YWALLS>(L, odd_next, out, st); break;
    default: launch_export_g<S, GEOM_TUBE>(L, odd_next, out, st); break;
  }
}
}  // namespace

void launch_collide(const LatticeDev& L, const RowInfo* rows, int n_rows, int storage, bool odd, bool dense, bool early,
                    cudaStream_t st) {
  if (n_rows == 0) return;
  switch (storage) {
    case STORE_F32: launch_collide_s<STORE_F32>(L, rows, n_rows, odd, dense, early, st); break;
    case STORE_F16: launch_collide_s<STORE_F16>(L, rows, n_rows, odd, dense, early, st); break;
    default: launch_collide_s<STORE_BF16>(L, rows, n_rows, odd, dense, early, st); break;
  }
}

void launch_init_equilibrium(const LatticeDev& L, int storage, cudaStream_t st) {
  switch (storage) {
    case STORE_F32: launch_init_s<STORE_F32>(L, st); break;
    case STORE_F16: launch_init_s<STORE_F16>(L, st); break;
    default: launch_init_s<STORE_BF16>(L, st); break;
  }
}

void launch_export(const LatticeDev& L, int storage, bool odd_next, double* out, cudaStream_t st) {
  switch (storage) {
    case STORE_F32: launch_export_s<STORE_F32>(L, odd_next, out, st); break;
    case STORE_F16: launch_export_s<STORE_F16>(L, odd_next, out, st); break;
    default: launch_export_s<STORE_BF16>(L, odd_next, out, st); break;
  }
}

void launch_import(const LatticeDev& L, int storage, const double* in, cudaStream_t st) {
  switch (storage) {
    case STORE_F32: k_import<STORE_F32><<<blocks_for(L.N), 256, 0, st>>>(L, in); break;
    case STORE_F16: k_import<STORE_F16><<<blocks_for(L.N), 256, 0, st>>>(L, in); break;
    default: k_import<STORE_BF16><<<blocks_for(L.N), 256, 0, st>>>(L, in); break;
  }
}

void launch_set_moments(const LatticeDev& L, const double* rho, const double* u, cudaStream_t st) {
  k_set_moments<<<blocks_for(L.N), 256, 0, st>>>(L, rho, u);
}

void launch_get_moments(const LatticeDev& L, double* rho, double* u, cudaStream_t st) {
  k_get_moments<<<blocks_for(L.N), 256, 0, st>>>(L, rho, u);
}

void launch_diagnostics(const LatticeDev& L, const RowInfo* rows, int n_rows, double* out, unsigned* umax2_bits,
                        cudaStream_t st) {
  const unsigned n = (unsigned)((long long)n_rows * L.nx);  // at most N, below 2^31
  if (n == 0) return;
  const int rounds = n >= 1216u * (2 * DIAG_LOADS * 256) ? 2 : 1;
  const unsigned span = (unsigned)rounds * DIAG_LOADS * 256, blocks = (n + span - 1) / span;
  k_diagnostics<<<blocks < 1216u ? blocks : 1216u, 256, 0, st>>>(L, rows, n, rounds, out, umax2_bits);
}

}  // namespace ibm
