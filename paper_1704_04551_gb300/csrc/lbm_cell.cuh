// Device-side bodies of the lattice-Boltzmann kernels, shared by the
// single-lattice kernels (lbm.cu) and the batched serving kernels
// (serve.cu). Method: Sec. 2.1 of arXiv:1704.04551 — Eq. lbm (stream + BGK
// collide + force term), Eq. BGKequilibrium, Eq. rho_u (moments with the
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
#pragma once
#include "common.cuh"

namespace ibm {

namespace lbm_detail {

template <int S>
struct Pop {
  using St = Store<S>;
  using T = typename St::T;
  __device__ static __forceinline__ float ld(const T* p, int i) {
    if constexpr (S == STORE_F32) return *p;
    else if constexpr (S == STORE_F16) return __half2float(*p) * (1.0f / dev_scale(i));
    else return __bfloat162float(*p) * (1.0f / dev_scale(i));
  }
  __device__ static __forceinline__ void st(T* p, int i, float v) {
    if constexpr (S == STORE_F32) *p = v;
    else if constexpr (S == STORE_F16) *p = __float2half_rn(v * dev_scale(i));
    else *p = __float2bfloat16_rn(v * dev_scale(i));
  }
  // the stored value itself (K_i d_i for the half-precision formats)
  __device__ static __forceinline__ float ld_raw(const T* p) {
    if constexpr (S == STORE_F32) return *p;
    else if constexpr (S == STORE_F16) return __half2float(*p);
    else return __bfloat162float(*p);
  }
  __device__ static __forceinline__ void st_raw(T* p, float v) {
    if constexpr (S == STORE_F32) *p = v;
    else if constexpr (S == STORE_F16) *p = __float2half_rn(v);
    else *p = __float2bfloat16_rn(v);
  }
};

struct Cell {
  int x, y, z;
  unsigned smask;          // bit (cy+1)*3 + (cz+1): neighbour in that (y,z) direction is solid
  int oxp, oxm, oyp, oym, ozp, ozm;  // wrapped element offsets of the six axis neighbours
};

template <int GEOM>
__device__ __forceinline__ bool make_cell(const LatticeDev& L, int idx, Cell& c) {
  const int nx = L.nx, ny = L.ny, nz = L.nz;
  c.x = idx % nx;
  const int t = idx / nx;
  c.y = t % ny;
  c.z = t / ny;
  c.smask = 0u;
  if constexpr (GEOM != GEOM_PERIODIC) {
    if (solid_yz(L, c.y, c.z)) return false;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
      for (int dz = -1; dz <= 1; ++dz)
        if (solid_yz(L, c.y + dy, c.z + dz)) c.smask |= 1u << ((dy + 1) * 3 + (dz + 1));
  }
  c.oxp = (c.x == nx - 1) ? -(nx - 1) : 1;
  c.oxm = (c.x == 0) ? (nx - 1) : -1;
  const int sy = nx, sz = nx * ny;
  c.oyp = (c.y == ny - 1) ? -(ny - 1) * sy : sy;
  c.oym = (c.y == 0) ? (ny - 1) * sy : -sy;
  c.ozp = (c.z == nz - 1) ? -(nz - 1) * sz : sz;
  c.ozm = (c.z == 0) ? (nz - 1) * sz : -sz;
  return true;
}

// element offset of the neighbour x + s*c_i
__device__ __forceinline__ int nb_off(const Cell& c, int i, int s) {
  const int dx = s * cx(i), dy = s * cy(i), dz = s * cz(i);
  return (dx > 0 ? c.oxp : (dx < 0 ? c.oxm : 0)) + (dy > 0 ? c.oyp : (dy < 0 ? c.oym : 0)) +
         (dz > 0 ? c.ozp : (dz < 0 ? c.ozm : 0));
}
// is x + s*c_i solid?
__device__ __forceinline__ bool nb_solid(const Cell& c, int i, int s) {
  return (c.smask >> ((s * cy(i) + 1) * 3 + (s * cz(i) + 1))) & 1u;
}

}  // namespace lbm_detail
using namespace lbm_detail;

// Collision of one cell (Eqs. rho_u, BGKequilibrium, the Guo term) on its
// 19 loaded values d (in place; the stored values K_i d_i for the
// half-precision formats): moments with the half-force shift (the force
// density is read where the cell's tile is touched, and the moments are
// written there or everywhere with DENSE), BGK relaxation and the Guo term.
// Returns rho (for the moving-wall term of the streaming).
template <int S, bool DENSE>
__device__ __forceinline__ float relax_cell(const LatticeDev& L, float d[Q], int idx, int tile) {
  // HALF: d[] holds the stored values K_i d_i of the half-precision formats
  // (K_i = dev_scale(i), a power of two, so that folding 1/K_i into the
  // moment sums and K_i into the update constants is exact).
  constexpr bool HALF = S != STORE_F32;
  // moments (Eq. rho_u): rho = sum f, rho u = sum f c + g/2
  float drho = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float k = HALF ? 1.0f / dev_scale(i) : 1.0f;
    drho = fmaf(d[i], k, drho);
    if (cx(i)) jx = fmaf(d[i], cx(i) * k, jx);
    if (cy(i)) jy = fmaf(d[i], cy(i) * k, jy);
    if (cz(i)) jz = fmaf(d[i], cz(i) * k, jz);
  }
  float Gx = L.g0x, Gy = L.g0y, Gz = L.g0z;
  const bool touched = L.flags[tile] != 0;
  if (touched) {
    const float4 gg = L.g[idx];
    Gx += gg.x; Gy += gg.y; Gz += gg.z;
  }
  const float rho = 1.0f + drho;
  const float irho = 1.0f / rho;
  const float ux = (jx + 0.5f * Gx) * irho;
  const float uy = (jy + 0.5f * Gy) * irho;
  const float uz = (jz + 0.5f * Gz) * irho;
  if (DENSE || touched) L.uw[idx] = make_float4(ux, uy, uz, drho);

  // BGK relaxation toward the equilibrium (Eq. BGKequilibrium) plus the Guo
  // term. Written per direction: a form that shares the parts of opposite
  // directions (c_{i+1} = -c_i) saves a few percent of the collide time but
  // doubled the FP32 velocity error against the FP64 oracle after 1000
  // coupled steps of the red-cell tube (1.8e-5 vs 9.4e-6, measured).
  const float om = L.omega, pre = L.guo_pre;
  const float usq15 = 1.5f * (ux * ux + uy * uy + uz * uz);
  const float uG = ux * Gx + uy * Gy + uz * Gz;
  if constexpr (!HALF) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const float w = wgt(i);
      const float cu = cx(i) * ux + cy(i) * uy + cz(i) * uz;
      const float cG = cx(i) * Gx + cy(i) * Gy + cz(i) * Gz;
      const float deq = w * (drho + rho * (3.0f * cu + 4.5f * cu * cu - usq15));
      const float Fi = pre * w * (3.0f * (cG - uG) + 9.0f * cu * cG);
      d[i] = d[i] + om * (deq - d[i]) + Fi;
    }
  } else {
    // The same update, regrouped for the half-precision formats (their
    // rounding dominates the error): with cu = c.u and cG = c.G,
    //   K_i (om f^eq_i + F_i) = K_i w_i [T0 + cu (3 om rho + 4.5 om rho cu + 9 pre cG) + 3 pre cG],
    //   T0 = om (drho - rho 1.5 u^2) - 3 pre u.G,
    // K_i w_i = 8/9 for every moving direction (4/3 at rest), and the pair
    // i, i+1 = opp(i) shares the even part in cu and flips the odd part.
    const float om1 = 1.0f - om;
    const float T0 = om * (drho - rho * usq15) - 3.0f * pre * uG;
    constexpr float KW = 8.0f / 9.0f;
    const float A = (KW * 3.0f) * om * rho, B = (KW * 4.5f) * om * rho;
    const float P3 = (KW * 3.0f) * pre, P9 = (KW * 9.0f) * pre;
    const float T0w = KW * T0;
    d[0] = fmaf(om1, d[0], (4.0f / 3.0f) * T0);
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const float cu = cx(i) * ux + cy(i) * uy + cz(i) * uz;
      const float cG = cx(i) * Gx + cy(i) * Gy + cz(i) * Gz;
      const float even = fmaf(fmaf(B, cu, P9 * cG), cu, T0w);
      const float odd = fmaf(A, cu, P3 * cG);
      d[i] = fmaf(om1, d[i], even + odd);
      d[i + 1] = fmaf(om1, d[i + 1], even - odd);
    }
  }

  return rho;
}

// One fluid cell of the fused collide-stream-force step (x in the row R).
// IDX32: element offsets of the neighbour-addressed (odd) step computed in
// 32 bits, valid while 19 N < 2^32 (fewer integer instructions than 64-bit
// address arithmetic per population; the odd step is issue-bound).
// INTERIOR: the row's y/z neighbour rows are all fluid (R.smask == 0), so
// no population is bounced back and the solid tests drop out.
template <int S, int ODD, int GEOM, bool DENSE, bool IDX32 = false, bool INTERIOR = false>
__device__ __forceinline__ void collide_cell(const LatticeDev& L, const RowInfo& R, int x) {
  constexpr bool WALLS = GEOM != GEOM_PERIODIC && !INTERIOR;  // solid neighbours possible
  using P = Pop<S>;
  using T = typename P::T;
  const int idx = R.base + x;
  Cell c;
  c.x = x;
  c.y = R.y;
  c.smask = (unsigned)R.smask;
  c.oxp = (x == L.nx - 1) ? 1 - L.nx : 1;
  c.oxm = (x == 0) ? L.nx - 1 : -1;
  c.oyp = R.oyp; c.oym = R.oym; c.ozp = R.ozp; c.ozm = R.ozm;
  T* A = reinterpret_cast<T*>(L.pop);
  const size_t N = (size_t)L.N;

  // f_j(x) sits at A[x][j] (even step) or at A[x - c_j][opp(j)] (odd step;
  // A[x][j] if x - c_j is solid). In both parities f*_i(x) goes back to the
  // slot that held f_opp(i)(x), which covers streaming and half-way
  // bounce-back alike.
  // element offset of population j at cell e (32- or 64-bit arithmetic)
  auto elem = [&](int j, int e) -> const T* {
    if constexpr (IDX32) return A + (unsigned)((unsigned)j * (unsigned)N + (unsigned)e);
    else return A + (size_t)j * N + e;
  };
  constexpr bool HALF = S != STORE_F32;  // d[] holds K_i d_i (see relax_cell)
  float d[Q];
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    if (!ODD || j == 0 || (WALLS && nb_solid(c, j, -1)))
      d[j] = P::ld_raw(elem(j, idx));
    else
      d[j] = P::ld_raw(elem(opp(j), idx + nb_off(c, j, -1)));
  }

  const float rho = relax_cell<S, DENSE>(L, d, idx, R.trow + (x >> TILE_X_SHIFT));

  // Recompute the write addresses from a few laundered registers instead of
  // keeping the 19 read addresses alive across the collision (which spills).
  int widx = idx;
  asm volatile("" : "+r"(widx), "+r"(c.oxp), "+r"(c.oxm), "+r"(c.oyp), "+r"(c.oym), "+r"(c.ozp), "+r"(c.ozm),
               "+r"(c.smask));
  // streaming with half-way bounce-back (moving-wall term on y walls)
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    float v = d[i];
    const bool sol = WALLS && i != 0 && nb_solid(c, i, +1);
    if (GEOM == GEOM_YWALLS && sol && cx(i) != 0) {
      // stored into slot opp(i): the half-precision scale of that slot
      const float uw = (c.y + cy(i) < 0) ? L.wall_u0 : L.wall_u1;
      v -= (HALF ? dev_scale(opp(i)) : 1.0f) * 6.0f * wgt(i) * rho * (float)cx(i) * uw;
    }
    if (!ODD || i == 0 || sol)
      P::st_raw(const_cast<T*>(elem(opp(i), widx)), v);
    else
      P::st_raw(const_cast<T*>(elem(i, widx + nb_off(c, i, +1))), v);
  }
}


// Two neighbouring fluid cells (x even, x + 1) in half-precision storage: 4-byte
// loads and stores (in the neighbour-addressed odd step, which takes rows
// without solid neighbours only, where a direction has no x component), and the
// arithmetic of
// relax_cell's half-precision branch in packed FP32 pairs. The single-cell
// kernel keeps ~48 KB of loads in flight on an SM, less than the memory's
// latency times its rate; a thread of this one has twice the bytes and half
// the instructions per cell. Needs an even nx (cell pairs aligned to 4 bytes).
template <int S, int ODD, int GEOM, bool DENSE, bool IDX32 = false>
__device__ __forceinline__ void collide_pair(const LatticeDev& L, const RowInfo& R, int x) {
  static_assert(S != STORE_F32, "half-precision storage");
  using P = Pop<S>;
  using T = typename P::T;
  T* A = reinterpret_cast<T*>(L.pop);
  const int idx = R.base + x;
  const size_t N = (size_t)L.N;
  auto elem = [&](int j, int e) -> T* {
    if constexpr (IDX32) return A + (unsigned)((unsigned)j * (unsigned)N + (unsigned)e);
    else return A + (size_t)j * N + e;
  };
  // odd step: element offset of the pair's row along s c_i, and of its two
  // cells there (periodic x)
  int oyp = R.oyp, oym = R.oym, ozp = R.ozp, ozm = R.ozm;
  int left = x == 0 ? L.nx - 1 : -1, right = x + 2 == L.nx ? 2 - L.nx : 2;  // to x - 1, x + 2
  auto row_off = [&](int i, int s) {
    const int dy = s * cy(i), dz = s * cz(i);
    return (dy > 0 ? oyp : (dy < 0 ? oym : 0)) + (dz > 0 ? ozp : (dz < 0 ? ozm : 0));
  };
  F32x2 d[Q];
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    if (ODD && cx(j) != 0) {  // f_j(x) is at x - c_j
      const int e = idx + row_off(j, -1);
      d[j] = cx(j) > 0 ? pack2(P::ld_raw(elem(opp(j), e + left)), P::ld_raw(elem(opp(j), e)))
                       : pack2(P::ld_raw(elem(opp(j), e + 1)), P::ld_raw(elem(opp(j), e + right)));
      continue;
    }
    const unsigned w = *reinterpret_cast<const unsigned*>(ODD ? elem(opp(j), idx + row_off(j, -1)) : elem(j, idx));
    if constexpr (S == STORE_F16) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w));
      d[j] = pack2(f.x, f.y);
    } else {
      d[j] = pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
  }
  F32x2 drho = both(0.f), jx = both(0.f), jy = both(0.f), jz = both(0.f);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float k = 1.0f / dev_scale(i);
    drho = fma2(d[i], both(k), drho);
    if (cx(i)) jx = fma2(d[i], both(cx(i) * k), jx);
    if (cy(i)) jy = fma2(d[i], both(cy(i) * k), jy);
    if (cz(i)) jz = fma2(d[i], both(cz(i) * k), jz);
  }
  F32x2 Gx = both(L.g0x), Gy = both(L.g0y), Gz = both(L.g0z);
  const bool touched = L.flags[R.trow + (x >> TILE_X_SHIFT)] != 0;  // (a tile holds both cells)
  if (touched) {
    const float4 a = L.g[idx], b = L.g[idx + 1];
    Gx = add2(Gx, pack2(a.x, b.x));
    Gy = add2(Gy, pack2(a.y, b.y));
    Gz = add2(Gz, pack2(a.z, b.z));
  }
  const F32x2 rho = add2(both(1.0f), drho);
  float r0, r1;
  unpack2(rho, r0, r1);
  const F32x2 irho = pack2(1.0f / r0, 1.0f / r1);
  const F32x2 ux = mul2(fma2(both(0.5f), Gx, jx), irho);
  const F32x2 uy = mul2(fma2(both(0.5f), Gy, jy), irho);
  const F32x2 uz = mul2(fma2(both(0.5f), Gz, jz), irho);
  if (DENSE || touched) {
    float x0, x1, y0, y1, z0, z1, e0, e1;
    unpack2(ux, x0, x1);
    unpack2(uy, y0, y1);
    unpack2(uz, z0, z1);
    unpack2(drho, e0, e1);
    L.uw[idx] = make_float4(x0, y0, z0, e0);
    L.uw[idx + 1] = make_float4(x1, y1, z1, e1);
  }
  const float om = L.omega, pre = L.guo_pre;
  constexpr float KW = 8.0f / 9.0f;
  const F32x2 usq15 = mul2(both(1.5f), fma2(uz, uz, fma2(uy, uy, mul2(ux, ux))));
  const F32x2 uG = fma2(uz, Gz, fma2(uy, Gy, mul2(ux, Gx)));
  const F32x2 om1 = both(1.0f - om);
  const F32x2 T0 = sub2(mul2(both(om), sub2(drho, mul2(rho, usq15))), mul2(both(3.0f * pre), uG));
  const F32x2 Aq = mul2(both((KW * 3.0f) * om), rho), Bq = mul2(both((KW * 4.5f) * om), rho);
  const F32x2 P3 = both((KW * 3.0f) * pre), P9 = both((KW * 9.0f) * pre);
  const F32x2 T0w = mul2(both(KW), T0);
  // component of a direction along +-(c_x, c_y, c_z)
  auto along = [](int i, F32x2 a, F32x2 b, F32x2 c) {
    F32x2 s = both(0.f);
    bool have = false;
    auto take = [&](int k, F32x2 v) {
      if (k == 0) return;
      s = have ? (k > 0 ? add2(s, v) : sub2(s, v)) : (k > 0 ? v : mul2(both(-1.0f), v));
      have = true;
    };
    take(cx(i), a);
    take(cy(i), b);
    take(cz(i), c);
    return s;
  };
  // (write addresses recomputed, not kept across the collision)
  int widx = idx;
  asm volatile("" : "+r"(widx), "+r"(left), "+r"(right), "+r"(oyp), "+r"(oym), "+r"(ozp), "+r"(ozm));
  auto store = [&](int i, F32x2 v) {  // f*_i of both cells
    float a, b;
    unpack2(v, a, b);
    if (ODD && cx(i) != 0) {
      const int e = widx + row_off(i, +1);
      P::st_raw(elem(i, cx(i) > 0 ? e + 1 : e + left), a);
      P::st_raw(elem(i, cx(i) > 0 ? e + right : e), b);
      return;
    }
    unsigned w;
    if constexpr (S == STORE_F16) {
      const __half2 p = __floats2half2_rn(a, b);
      w = *reinterpret_cast<const unsigned*>(&p);
    } else {
      const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
      w = *reinterpret_cast<const unsigned*>(&p);
    }
    *reinterpret_cast<unsigned*>(ODD ? elem(i, widx + row_off(i, +1)) : elem(opp(i), widx)) = w;
  };
  store(0, fma2(om1, d[0], mul2(both(4.0f / 3.0f), T0)));
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const F32x2 cu = along(i, ux, uy, uz), cG = along(i, Gx, Gy, Gz);
    const F32x2 even = fma2(fma2(Bq, cu, mul2(P9, cG)), cu, T0w);
    const F32x2 odd = fma2(Aq, cu, mul2(P3, cG));
    F32x2 p = fma2(om1, d[i], add2(even, odd)), m = fma2(om1, d[i + 1], sub2(even, odd));
    if (!ODD && GEOM == GEOM_YWALLS && cx(i) != 0 && cy(i) != 0) {
      // half-way bounce-back at the moving walls, as in collide_cell
      auto wall = [&](int k, F32x2 v) {
        const int yn = R.y + cy(k);
        if ((unsigned)yn < (unsigned)L.ny) return v;
        const float uw = yn < 0 ? L.wall_u0 : L.wall_u1;
        return fma2(both(-dev_scale(opp(k)) * 6.0f * wgt(k) * (float)cx(k) * uw), rho, v);
      };
      p = wall(i, p);
      m = wall(i + 1, m);
    }
    store(i, p);
    store(i + 1, m);
  }
}

}  // namespace ibm
