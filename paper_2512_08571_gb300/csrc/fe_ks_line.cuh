// Default cell kernel: one line per thread, three shared tiles, (cell, column)
// pairs flattened into tiles.
//
// Paper: Algorithm 2 called from Algorithm 1, as in fe_ks_local.cuh, with the
// sweeps ordered and fused so that a point costs 23 shared-memory accesses and
// a tile eight block barriers (27 and nine for the kernels there):
//   a  z lines of nodes:    gather X, N_z                                  -> A
//   b  y lines:             N_y                                            -> A
//   c  x lines:             N_x -> Y0, D~_x Y0                             -> A, B
//   d  y lines:             D~_y Y0                                        -> C
//   e  z lines:             D~_z, quadrature-point step, Z + D~_z^T W_z    -> A; W_x, W_y -> B, C
//   f  y lines:             A + D~_y^T W_y                                 -> A
//   g  x lines:             N_x^T (A + D~_x^T W_x)                         -> A
//   h  y lines:             N_y^T                                          -> A
//   i  z lines of nodes:    N_z^T, expansion F Delta P, assembly
// The node lines of a and i are z lines, so the lanes of a warp read consecutive
// nodes of the DoF list and of F, and the Gauss lines of e consecutive points of
// the coefficients.  A thread reads its own line of A in i and overwrites it in
// the next tile's a, so no barrier separates two tiles.
//
// Two forms.  WIDE (FP32, n_q <= 9, at least a tile of columns): a block walks the
// column tiles of one cell and keeps the cell's coefficients, DoF list and
// destinations in shared memory (phase e waited for them for 40 % of its time when
// they came through the L1), and where they fit the next tile's rows of X arrive by
// cp.async behind phases b..i.  Otherwise the elements ("slots") of a tile are VG
// consecutive ones of the flattened [cell][column element] space, so a column count
// that is no multiple of the tile leaves no lane idle and a single vector (Lanczos)
// fills a tile with VG cells.  Blocks take every gridDim-th cell or tile: the cells
// that carry projectors are neighbours, and a contiguous share of them would make
// some blocks late.
//
// What bounds it.  FP64: the FP64 pipe (p = 6, 10^3 cells, 64 columns: 0.75 of 1.25 TFLOP/s,
// 5.15 -> 4.92 ms).  FP32: barriers and the latency of the shared-memory sweeps (p = 8:
// issue 54 % and FMA pipe 40 % busy with the 32 % of the warps that the three tiles and the staged tables
// leave room for); keeping lines in registers instead (a plane per thread, 12 accesses a point) takes
// 8 to 12 thousand straight-line instructions and was bound by the instruction cache, 11.8 ms
// against 6.4 of the kernels in fe_ks_local.cuh.  By colour there -> here: p = 8, 16^3 cells, 256
// columns, 19 atoms 7.6 -> 6.6 ms; complex p = 7, 10^3, 64 columns 1.70 -> 0.65 ms; n_q = 11, 8^3,
// 32 columns 565 -> 235 us; p = 6, 12^3, 37 columns 706 -> 333 us; FP64 p = 4, 4^3, 8 columns
// 223 -> 24.6 us.  Wide / flat form at p = 8, 16^3, 256
// columns without atoms: 5.3 / 5.7 ms.
//
// Elements: every type works on 8-byte elements -- two FP32 columns (packed FP32x2
// instructions; the re and im columns of a complex vector), one FP64 column, or
// one column in a pair of floats (fe_ks_line_ff.cuh).
#pragma once
#include "fe_ks_local.cuh"

namespace feks {

// ---- elements

__device__ __forceinline__ f2v& operator+=(f2v& a, f2v b) {
  a = a + b;
  return a;
}
__device__ __forceinline__ f2v operator*(f2v a, f2v b) {
  f2v r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2v fma(f2v a, f2v b, f2v c) {
  f2v r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// T: arithmetic type of the tables and coefficients, TS: storage type of X, Y, Q
template <typename T, typename TS>
struct Elem {   // FP64 and pairs of floats: one column
  using V = T;
  static constexpr int CPE = 1;   // columns per element
  static __device__ __forceinline__ V load(const TS* p, bool, bool) { return Num<T>::in(__ldg(p)); }
  static __device__ __forceinline__ TS stored(V v) {
    if constexpr (std::is_same<T, ff2>::value)
      return f2d_bits(v.hi) + f2d_bits(v.lo);
    else
      return v;
  }
  static __device__ __forceinline__ void store(TS* p, V v, bool, bool, bool accum) {
    TS s = stored(v);
    if (accum) s += *p;
    *p = s;
  }
  static __device__ __forceinline__ void add(TS* p, V v, bool, bool) {
    atomicAdd(p, stored(v));
  }
  // -i (a + i b) = b - i a: the re column adds the partner's im, the im column subtracts its re
  static __device__ __forceinline__ V minus_i(V kk, int v, unsigned mask) {
    V kp;
    if constexpr (std::is_same<T, ff2>::value)
      kp = ff_make(__shfl_xor_sync(mask, kk.hi, 1), __shfl_xor_sync(mask, kk.lo, 1));
    else
      kp = __shfl_xor_sync(mask, kk, 1);
    return (v & 1) ? -kp : kp;
  }
};
template <>
struct Elem<float, float> {   // two FP32 columns
  using V = f2v;
  static constexpr int CPE = 2;
  // vec: 8-byte access; two: the second column exists
  static __device__ __forceinline__ V load(const float* p, bool vec, bool two) {
    if (vec) {
      V r;
      r.v = __ldg(reinterpret_cast<const unsigned long long*>(p));
      return r;
    }
    return f2v_make(__ldg(p), two ? __ldg(p + 1) : 0.f);
  }
  static __device__ __forceinline__ void store(float* p, V v, bool vec, bool two, bool accum) {
    if (vec) {
      if (accum) {
        V o;
        o.v = *reinterpret_cast<const unsigned long long*>(p);
        v = v + o;
      }
      *reinterpret_cast<unsigned long long*>(p) = v.v;
    } else {
      const float2 s = f2v_split(v);
      p[0] = accum ? p[0] + s.x : s.x;
      if (two) p[1] = accum ? p[1] + s.y : s.y;
    }
  }
  static __device__ __forceinline__ void add(float* p, V v, bool vec, bool two) {
    const float2 s = f2v_split(v);
    if (vec) {
      asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(s.x), "f"(s.y) : "memory");
    } else {
      atomicAdd(p, s.x);
      if (two) atomicAdd(p + 1, s.y);
    }
  }
  static __device__ __forceinline__ V minus_i(V kk, int, unsigned) {
    const float2 s = f2v_split(kk);
    return f2v_make(s.y, -s.x);
  }
};

template <typename V>
__device__ __forceinline__ V elem_zero() {
  if constexpr (std::is_same<V, f2v>::value)
    return f2v_make(0.f, 0.f);
  else
    return Num<V>::zero();
}

// The 1D tables in the element type: FP32 entries twice, so that a packed
// instruction takes its 64-bit coefficient from the constant bank.
template <typename T, typename TS>
struct LineParams : LocalParams<T, TS> {};
template <>
struct LineParams<float, float> : LocalParams<float, float> {
  EOTables<f2v> tab2;
  int run;   // wide form: column tiles of a cell per unit of work
};
template <typename T, typename TS>
__device__ __forceinline__ const auto& line_tables(const LineParams<T, TS>& p) {
  if constexpr (std::is_same<T, float>::value)
    return p.tab2;
  else
    return p.tab;
}

// ---- shape

// Elements per tile, block size and resident blocks per SM for n_q points: n_q^2 VG
// threads near a multiple of 32, three tiles of shared memory per block, and a
// register budget (65536 / (MINB NT)) that holds phase e's three lines.  VG is a
// power of two so that, with the odd y pitch PY, the 16 lanes of a shared-memory
// phase fall into different banks in every direction.  SMALL: tiles of two elements (a
// complex pair), for launches whose full tiles would leave multiprocessors without one.
constexpr int line_vg(int nq, bool small) { return small ? 2 : nq >= 11 ? 2 : nq >= 7 ? 4 : nq >= 5 ? 8 : 16; }
constexpr int line_minb(int nq, bool small, int nt) {
  return small ? (768 / nt < 16 ? 768 / nt : 16)
               : nq == 11 ? 3 : nq == 10 || nq == 9 ? 2 : nq == 8 || nq == 7 ? 3 : nq == 6 ? 2 : nq == 5 ? 3 : nq == 4 ? 2 : 4;
}
template <int NQ, bool SMALL = false>
struct LineShape {
  static constexpr int VG = line_vg(NQ, SMALL);
  static constexpr int NT = (NQ * NQ * VG + 31) / 32 * 32;
  static constexpr int MINB = line_minb(NQ, SMALL, NT);
  static constexpr int PY = NQ | 1;
  static constexpr int SX = VG, SY = PY * VG, SZ = NQ * SY, BUF = NQ * SZ;
  static constexpr size_t tiles = 3 * (size_t)BUF * 8;
};

// Forms of the kernel
enum : int { kLineFlat = 0, kLineWide = 1, kLineSmall = 2 };

// Whether tiles of two elements give the fullest multiprocessor clearly (an eighth) less to do
// than full ones: 64 cells of 8 FP64 columns at p = 4 took 31.8 us on 64 full tiles, 24.6 us on 256
// of these; once every multiprocessor has several tiles the full ones' vector width wins.  VG, VS:
// elements of a full and of a small tile; M: small ones are taken up to M eighths of the full ones' work
template <int VG, int VS, int M = 7>
bool line_small(int64_t slots, int sms) {
  const int64_t full = ((slots + VG - 1) / VG + sms - 1) / sms * VG, small = ((slots + VS - 1) / VS + sms - 1) / sms * VS;
  return 8 * small <= M * full;
}

// Shared memory of the wide form after the three tiles: [coefficients] [DoFs] [destinations] [a pair's
// projections Q of the tile's columns] [X tile].  A pair's F block takes tiles B and C, free in h and i.
constexpr int kLineMaxProj = 16;   // projectors an atom can carry
template <int NP, int NQ, bool CPLX, bool BOX>
struct WideShape {
  using S = LineShape<NQ>;
  static constexpr int NP3 = NP * NP * NP, NQ3 = NQ * NQ * NQ;
  static constexpr int NCF = BOX ? 4 : CPLX ? kCoefCplx : kCoefReal;   // coefficient rows kept (BOX: V_L, V_G)
  static constexpr size_t cf = ((size_t)NCF * NQ3 * 4 + 15) / 16 * 16, idx = ((size_t)NP3 * 4 + 15) / 16 * 16;
  static constexpr size_t xs = (size_t)NP3 * S::VG * 8;
  static constexpr size_t qs = (size_t)kLineMaxProj * S::VG * 8;
  static constexpr size_t rest = S::tiles + cf + 2 * idx + qs;
  static constexpr bool STAGE_X = (rest + xs + 1024) * S::MINB <= 228 * 1024;
  static constexpr size_t bytes = rest + (STAGE_X ? xs : 0);
  static constexpr int MINB = (bytes + 1024) * S::MINB <= 228 * 1024 ? S::MINB : S::MINB - 1;
};

template <int NP, int NQ, bool CPLX, bool BOX, int FORM>
constexpr int line_blocks() {
  if constexpr (FORM == kLineWide)
    return WideShape<NP, NQ, CPLX, BOX>::MINB;
  else
    return LineShape<NQ, FORM == kLineSmall>::MINB;
}

template <typename T, typename TS, int NP, int NQ, bool CPLX, bool BOX, int FORM>
__global__ void __launch_bounds__(LineShape<NQ, FORM == kLineSmall>::NT, line_blocks<NP, NQ, CPLX, BOX, FORM>())
    fe_line_kernel(const __grid_constant__ LineParams<T, TS> p) {
  constexpr bool WIDE = FORM == kLineWide;
  using S = LineShape<NQ, FORM == kLineSmall>;
  using E = Elem<T, TS>;
  using V = typename E::V;
  constexpr int VG = S::VG, SX = S::SX, SY = S::SY, SZ = S::SZ, NQ2 = NQ * NQ, NQ3 = NQ * NQ2, NP2 = NP * NP;
  constexpr int NP3 = NP * NP2, CPE = E::CPE, NT = S::NT;
  using W = WideShape<NP, NQ, CPLX, BOX>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const auto& tab = line_tables(p);
  const int v = threadIdx.x % VG, ln = threadIdx.x / VG;
  V* const A = reinterpret_cast<V*>(smem_raw) + v;
  V* const B = A + S::BUF;
  V* const C = B + S::BUF;
  [[maybe_unused]] float* const cfs = reinterpret_cast<float*>(smem_raw + S::tiles);
  [[maybe_unused]] int* const sdof = reinterpret_cast<int*>(smem_raw + S::tiles + W::cf);
  [[maybe_unused]] int* const sdst = reinterpret_cast<int*>(smem_raw + S::tiles + W::cf + W::idx);
  [[maybe_unused]] float* const qs = reinterpret_cast<float*>(smem_raw + S::tiles + W::cf + 2 * W::idx);
  [[maybe_unused]] float* const Fs = reinterpret_cast<float*>(smem_raw + (size_t)S::BUF * 8);
  constexpr int CW = CPLX ? 2 : 1;
  // wide form: a pair's F block fits tiles B and C
  [[maybe_unused]] const bool fits_f = (size_t)p.n_proj * NP3 * CW * sizeof(float) <= 2 * (size_t)S::BUF * 8;
  [[maybe_unused]] int pbeg = 0, pend = 0, pair0 = 0, atom0 = 0;   // wide form: the cell's pairs, its first one
  [[maybe_unused]] V* const XS = reinterpret_cast<V*>(smem_raw + W::rest);
  const bool node_line = ln < NP2, gauss_line = ln < NQ2, mixed_line = ln < NP * NQ;
  const unsigned gmask = CPLX ? __ballot_sync(0xffffffffu, gauss_line) : 0u;
  // this thread's lines: element offsets of Gauss lines along x, y, z and of node lines along z and y
  int ox = (ln % NQ) * SY + (ln / NQ) * SZ, oy = (ln % NQ) * SX + (ln / NQ) * SZ, oz = (ln % NQ) * SX + (ln / NQ) * SY;
  int on = (ln % NP) * SX + (ln / NP) * SY, om = (ln % NP) * SX + (ln / NP) * SZ;
  const bool vec = CPE == 1 || (p.ld % 2 == 0 && ((uintptr_t)p.X & 7) == 0);
  const bool vecq = CPE == 1 || (p.ld % 2 == 0 && ((uintptr_t)p.Q & 7) == 0);
  const bool vecy = CPE == 1 || (p.ld % 2 == 0 && ((uintptr_t)p.Y & 7) == 0);
  const int ncg = (p.ncols + CPE - 1) / CPE;   // column elements per cell

  // column elements [c0, c0 + VG) of the staged cell's rows of X -> XS (zero beyond ncols)
  [[maybe_unused]] auto stage_x = [&](int c0) {
    if constexpr (WIDE) {
      const bool v16 = p.ld % 4 == 0 && ((uintptr_t)p.X & 15) == 0;
      float* xs = reinterpret_cast<float*>(XS);
      if (v16) {
        constexpr int CH = VG / 2;
        for (int i = threadIdx.x; i < NP3 * CH; i += NT) {
          const int node = i / CH, col = c0 * 2 + (i % CH) * 4;
          int nb = (p.ncols - col) * 4;
          nb = nb < 0 ? 0 : nb > 16 ? 16 : nb;
          cp_async_16z(xs + i * 4, nb > 0 ? p.X + (int64_t)sdof[node] * p.ld + col : p.X, nb);
        }
      } else {
        for (int i = threadIdx.x; i < NP3 * VG * 2; i += NT) {
          const int node = i / (2 * VG), col = c0 * 2 + i % (2 * VG);
          const bool in = col < p.ncols;
          cp_async_4z(xs + i, in ? p.X + (int64_t)sdof[node] * p.ld + col : p.X, in ? 4 : 0);
        }
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
  };

  // a pair's F block -> B and C, and its projections of column elements [c0, c0 + VG) -> qs
  [[maybe_unused]] auto stage_f = [&](int pr, int atom, int c0) {
    if constexpr (WIDE) {
      const float* F = p.F + (int64_t)pr * p.n_proj * NP3 * CW;
      for (int i = threadIdx.x; i < p.n_proj * NP3 * CW; i += NT) cp_async_4(Fs + i, F + i);
      const float* Q = p.Q + (int64_t)atom * p.n_proj * p.ld;
      for (int i = threadIdx.x; i < p.n_proj * 2 * VG; i += NT) {
        const int col = 2 * c0 + i % (2 * VG);
        const bool in = col < p.ncols;
        cp_async_4z(qs + i, in ? Q + (int64_t)(i / (2 * VG)) * p.ld + col : Q, in ? 4 : 0);
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
  };

  // one tile: cell e, first column col of this lane; act: the lane stores; c0: the tile's first
  // column element (wide form).  next: called once phase a has read the tile's rows of X
  auto tile = [&](int e, int col, bool act, [[maybe_unused]] int c0, auto next) {
    const bool two = CPE == 1 || col + 1 < p.ncols;
    // a
    if (node_line) {
      V x[NP], y[NQ];
      const int* __restrict__ dofs = p.cell_dofs + (int64_t)e * NP3 + ln;
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const int d = WIDE ? sdof[ln + k * NP2] : dofs[k * NP2];
        if constexpr (WIDE && W::STAGE_X)
          x[k] = XS[(ln + k * NP2) * VG + v];
        else
          x[k] = E::load(p.X + (int64_t)d * p.ld + col, vec && two, two);
        if (p.dscale) x[k] = p.dscale[d] * x[k];
      }
      eo_apply<NP, NQ, 1>(x, y, tab.N);
#pragma unroll
      for (int q = 0; q < NQ; ++q) A[on + q * SZ] = y[q];
    }
    __syncthreads();
    next();
    // b
    if (mixed_line) {
      V x[NP], y[NQ];
#pragma unroll
      for (int j = 0; j < NP; ++j) x[j] = A[om + j * SY];
      eo_apply<NP, NQ, 1>(x, y, tab.N);
#pragma unroll
      for (int q = 0; q < NQ; ++q) A[om + q * SY] = y[q];
    }
    __syncthreads();
    // c
    if (gauss_line) {
      V x[NP], y[NQ], g[NQ];
#pragma unroll
      for (int i = 0; i < NP; ++i) x[i] = A[ox + i * SX];
      eo_apply<NP, NQ, 1>(x, y, tab.N);
#pragma unroll
      for (int q = 0; q < NQ; ++q) A[ox + q * SX] = y[q];
      eo_apply<NQ, NQ, -1>(y, g, tab.D);
#pragma unroll
      for (int q = 0; q < NQ; ++q) B[ox + q * SX] = g[q];
    }
    __syncthreads();
    // d
    if (gauss_line) {
      V x[NQ], g[NQ];
#pragma unroll
      for (int r = 0; r < NQ; ++r) x[r] = A[oy + r * SY];
      eo_apply<NQ, NQ, -1>(x, g, tab.D);
#pragma unroll
      for (int q = 0; q < NQ; ++q) C[oy + q * SY] = g[q];
    }
    __syncthreads();
    // e: Z = V^L Y0 + V^G.grad - i V^K.grad, W_s = sum_d G_sd grad_d + V^G_s Y0
    if (gauss_line) {
      V u[NQ], g[NQ], zc[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) u[q] = A[oz + q * SZ];
      eo_apply<NQ, NQ, -1>(u, g, tab.D);
      // coefficient row r of the point: cf[r NQ3] (BOX keeps rows 6..9 only)
      const T* cf;
      if constexpr (WIDE)
        cf = reinterpret_cast<const T*>(cfs) + ln - (BOX ? 6 * NQ3 : 0);
      else
        cf = p.coef + (int64_t)e * p.ncoef * NQ3 + ln;
      // axis-aligned cells: kinetic and Bloch coefficients are scalars of the cell times the point's
      // weight, formed in pairs so that they round once, as the stored ones do
      [[maybe_unused]] ff2 cs[3] = {}, ks[3] = {};
      if constexpr (BOX) {
        const ff2 w2 = ff_mul(ff_make(p.w[ln % NQ], p.wl[ln % NQ]), ff_make(p.w[ln / NQ], p.wl[ln / NQ]));
        const float* cc = p.cell_coef + 16 * (int64_t)e;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          cs[d] = ff_mul(ff_make(cc[d], cc[8 + d]), w2);
          if constexpr (CPLX) ks[d] = ff_mul(ff_make(cc[4 + d], cc[12 + d]), w2);
        }
      }
      [[maybe_unused]] auto weighted = [&](ff2 c, int q) -> float {
        return fmaf(c.hi, p.w[q], fmaf(c.hi, p.wl[q], c.lo * p.w[q]));
      };
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int s = oz + q * SZ;
        const T* cq = cf + q * NQ2;
        const V gx = B[s], gy = C[s], gz = g[q], uu = u[q];
        V z = T(cq[6 * NQ3]) * uu, w0, w1, w2;
        if constexpr (BOX) {
          w0 = weighted(cs[0], q) * gx;
          w1 = weighted(cs[1], q) * gy;
          w2 = weighted(cs[2], q) * gz;
        } else {
          const T G00 = cq[0], G01 = cq[NQ3], G02 = cq[2 * NQ3], G11 = cq[3 * NQ3], G12 = cq[4 * NQ3];
          const T G22 = cq[5 * NQ3];
          w0 = fma(G00, gx, fma(G01, gy, G02 * gz));
          w1 = fma(G01, gx, fma(G11, gy, G12 * gz));
          w2 = fma(G02, gx, fma(G12, gy, G22 * gz));
        }
        if (p.gga) {
          const T V0 = cq[7 * NQ3], V1 = cq[8 * NQ3], V2 = cq[9 * NQ3];
          z = fma(V0, gx, fma(V1, gy, fma(V2, gz, z)));
          w0 = fma(V0, uu, w0);
          w1 = fma(V1, uu, w1);
          w2 = fma(V2, uu, w2);
        }
        if constexpr (CPLX) {
          V kk;
          if constexpr (BOX) {
            kk = fma(weighted(ks[0], q), gx, fma(weighted(ks[1], q), gy, weighted(ks[2], q) * gz));
          } else {
            kk = fma(T(cq[10 * NQ3]), gx, fma(T(cq[11 * NQ3]), gy, T(cq[12 * NQ3]) * gz));
          }
          z += E::minus_i(kk, v, gmask);
        }
        B[s] = w0;
        C[s] = w1;
        u[q] = w2;
        zc[q] = z;
      }
      eo_apply<NQ, NQ, -1>(u, g, tab.Dt);
#pragma unroll
      for (int q = 0; q < NQ; ++q) A[oz + q * SZ] = zc[q] + g[q];
    }
    __syncthreads();
    // f
    if (gauss_line) {
      V x[NQ], g[NQ];
#pragma unroll
      for (int r = 0; r < NQ; ++r) x[r] = C[oy + r * SY];
      eo_apply<NQ, NQ, -1>(x, g, tab.Dt);
#pragma unroll
      for (int q = 0; q < NQ; ++q) A[oy + q * SY] = A[oy + q * SY] + g[q];
    }
    __syncthreads();
    // g
    if (gauss_line) {
      V x[NQ], g[NQ], y[NP];
#pragma unroll
      for (int r = 0; r < NQ; ++r) x[r] = B[ox + r * SX];
      eo_apply<NQ, NQ, -1>(x, g, tab.Dt);
#pragma unroll
      for (int q = 0; q < NQ; ++q) g[q] = A[ox + q * SX] + g[q];
      eo_apply<NQ, NP, 1>(g, y, tab.Nt);
#pragma unroll
      for (int i = 0; i < NP; ++i) A[ox + i * SX] = y[i];
    }
    __syncthreads();
    const bool staged_f = WIDE && pend > pbeg && fits_f;
    if (staged_f) stage_f(pair0, atom0, c0);   // arrives behind h
    // h
    if (mixed_line) {
      V x[NQ], y[NP];
#pragma unroll
      for (int q = 0; q < NQ; ++q) x[q] = A[om + q * SY];
      eo_apply<NQ, NP, 1>(x, y, tab.Nt);
#pragma unroll
      for (int j = 0; j < NP; ++j) A[om + j * SY] = y[j];
    }
    if (staged_f) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    // i
    V y[NP];
    if (node_line) {
      V x[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) x[q] = A[on + q * SZ];
      eo_apply<NQ, NP, 1>(x, y, tab.Nt);
    }
    if constexpr (WIDE) {
      if (staged_f)
        for (int pi = pbeg;;) {
          if (node_line) {
#pragma unroll 3
            for (int b = 0; b < p.n_proj; ++b) {
              V q;
              q.v = *reinterpret_cast<const unsigned long long*>(qs + (b * VG + v) * 2);
              if constexpr (!CPLX) {
#pragma unroll
                for (int k = 0; k < NP; ++k) y[k] = fma(Fs[b * NP3 + ln + k * NP2], q, y[k]);
              } else {
                const float2 s = f2v_split(q);
                const V iq = f2v_make(-s.y, s.x);
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                  const float2 f = *reinterpret_cast<const float2*>(Fs + (b * NP3 + ln + k * NP2) * 2);
                  y[k] = fma(f.x, q, fma(f.y, iq, y[k]));
                }
              }
            }
          }
          if (++pi >= pend) break;
          __syncthreads();   // the next pair of the cell takes the same place
          const int pr = p.cell_pairs[pi];
          stage_f(pr, p.pair_atom[pr], c0);
          asm volatile("cp.async.wait_group 0;\n" ::: "memory");
          __syncthreads();
        }
    }
    if (node_line && act) {
      if (p.cell_pair_ptr && !staged_f) {
        const int pb = p.cell_pair_ptr[e], pe = p.cell_pair_ptr[e + 1];
        for (int pi = pb; pi < pe; ++pi) {
          const int pr = p.cell_pairs[pi];
          const TS* Qa = p.Q + (int64_t)p.pair_atom[pr] * p.n_proj * p.ld;
          const T* __restrict__ Fp = p.F + ((int64_t)pr * p.n_proj * NP3 + ln) * (CPLX ? 2 : 1);
          // PB projectors at a time: their loads of Q and F are in flight together
          constexpr int PB = 3;
#pragma unroll 1
          for (int b0 = 0; b0 < p.n_proj; b0 += PB) {
            V q[PB], iq[PB];
#pragma unroll
            for (int u = 0; u < PB; ++u) {
              const TS* Qb = Qa + (int64_t)min(b0 + u, p.n_proj - 1) * p.ld + col;
              q[u] = E::load(Qb, vecq && two, two);
              if constexpr (CPLX) {
                // i (qr + i qi) = -qi + i qr
                if constexpr (CPE == 2) {
                  const float2 s = f2v_split(q[u]);
                  iq[u] = f2v_make(-s.y, s.x);
                } else {
                  const V qp = E::load(Qb - col + (col ^ 1), false, true);
                  iq[u] = (col & 1) ? qp : -qp;
                }
              }
            }
#pragma unroll
            for (int u = 0; u < PB; ++u) {
              if (b0 + u >= p.n_proj) break;
              const T* __restrict__ Fb = Fp + (int64_t)(b0 + u) * NP3 * (CPLX ? 2 : 1);
#pragma unroll
              for (int k = 0; k < NP; ++k) {
                if constexpr (CPLX)
                  y[k] = fma(Fb[k * NP2 * 2], q[u], fma(Fb[k * NP2 * 2 + 1], iq[u], y[k]));
                else
                  y[k] = fma(Fb[k * NP2], q[u], y[k]);
              }
            }
          }
        }
      }
      const int* __restrict__ dofs = p.cell_dofs + (int64_t)e * NP3 + ln;
      const bool vy = vecy && two;
      if (p.dst) {   // one launch for all cells: rows of one cell straight to Y, shared rows to their slots
        const int* __restrict__ dst = p.dst + (int64_t)e * NP3 + ln;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          V val = p.alpha * y[k];
          if (p.dscale) val = p.dscale[WIDE ? sdof[ln + k * NP2] : dofs[k * NP2]] * val;
          const int d = WIDE ? sdst[ln + k * NP2] : dst[k * NP2];
          if (d >= 0)
            E::store(p.Y + (int64_t)d * p.ld + col, val, vy, two, p.accum);
          else
            E::store(p.W + (int64_t)(~d) * p.ld + col, val, vy, two, false);
        }
      } else {       // one colour: no two cells of the launch share a row of Y
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          const int d = WIDE ? sdof[ln + k * NP2] : dofs[k * NP2];
          V val = p.alpha * y[k];
          if (p.dscale) val = p.dscale[d] * val;
          E::add(p.Y + (int64_t)d * p.ld + col, val, vy, two);
        }
      }
    }
  };

  if constexpr (WIDE) {
    // unit = (cell, run of its column tiles)
    const int ntile = (ncg + VG - 1) / VG, upc = (ntile + p.run - 1) / p.run;
    const int units = p.n_cells * upc;
    int staged = -1;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
      const int ci = u / upc, tb = (u - ci * upc) * p.run, te = min(ntile, tb + p.run);
      const int e = p.cells ? p.cells[ci] : ci;
      if (ci != staged) {
        __syncthreads();   // the last tile's readers of the staged tables are done
        for (int i = threadIdx.x; i < NP3; i += NT) {
          sdof[i] = p.cell_dofs[(int64_t)e * NP3 + i];
          if (p.dst) sdst[i] = p.dst[(int64_t)e * NP3 + i];
        }
        const T* g = p.coef + ((int64_t)e * p.ncoef + (BOX ? 6 : 0)) * NQ3;
        for (int i = threadIdx.x; i < W::NCF * NQ3; i += NT) cp_async_4(cfs + i, g + i);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        if (p.cell_pair_ptr) {
          pbeg = p.cell_pair_ptr[e], pend = p.cell_pair_ptr[e + 1];
          if (pend > pbeg) pair0 = p.cell_pairs[pbeg], atom0 = p.pair_atom[pair0];
        }
        staged = ci;
        __syncthreads();
      }
      if constexpr (W::STAGE_X) stage_x(tb * VG);
      for (int t = tb; t < te; ++t) {
        if (t == tb || W::STAGE_X) {
          asm volatile("cp.async.wait_group 0;\n" ::: "memory");
          __syncthreads();
        }
        const bool act = t * VG + v < ncg;
        tile(e, act ? (t * VG + v) * CPE : 0, act, t * VG, [&] {
          if constexpr (W::STAGE_X)
            if (t + 1 < te) stage_x((t + 1) * VG);
        });
      }
    }
  } else {
    const int64_t nslots = (int64_t)p.n_cells * ncg, ntiles = (nslots + VG - 1) / VG;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      // an idle lane repeats a slot of its own re/im parity and stores nothing
      const int64_t slot = t * VG + v;
      const bool act = slot < nslots;
      const int ci = act ? (int)(slot / ncg) : p.n_cells - 1;
      const int ce = act ? (int)(slot - (int64_t)ci * ncg) : (CPLX && CPE == 1) ? (int)(slot & 1) : 0;
      tile(p.cells ? p.cells[ci] : ci, ce * CPE, act, 0, [] {});
    }
  }
}

template <typename T, typename TS, int NP, int NQ, bool CPLX, bool BOX, int FORM>
cudaError_t launch_line_form(const Ctx& c, LineParams<T, TS>& lp, int64_t work, int sms, cudaStream_t s) {
  using S = LineShape<NQ, FORM == kLineSmall>;
  constexpr size_t bytes = FORM == kLineWide ? WideShape<NP, NQ, CPLX, BOX>::bytes : S::tiles;
  static bool attr_done[64] = {};
  const int dev = c.device & 63;
  auto k = fe_line_kernel<T, TS, NP, NQ, CPLX, BOX, FORM>;
  if (!attr_done[dev]) {
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (err != cudaSuccess) return err;
    attr_done[dev] = true;
  }
  const int64_t slots = (int64_t)line_blocks<NP, NQ, CPLX, BOX, FORM>() * sms;
  k<<<(int)(work < slots ? work : slots), S::NT, bytes, s>>>(lp);
  return cudaGetLastError();
}

template <typename T, typename TS, int NP, int NQ, bool CPLX, bool BOX>
cudaError_t launch_line_t(const Ctx& c, const LocalParams<T, TS>& prm, cudaStream_t s) {
  using S = LineShape<NQ>;
  constexpr int CPE = Elem<T, TS>::CPE;
  LineParams<T, TS> lp;
  static_cast<LocalParams<T, TS>&>(lp) = prm;
  if (prm.n_cells == 0) return cudaSuccess;
  const int ncg = (prm.ncols + CPE - 1) / CPE, sms = c.sms > 0 ? c.sms : 152;
  const int64_t elems = (int64_t)prm.n_cells * ncg;
  if constexpr (std::is_same<T, float>::value) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(&prm.tab);
    f2v* dst = reinterpret_cast<f2v*>(&lp.tab2);
    for (size_t i = 0; i < sizeof(prm.tab) / 4; ++i) dst[i].v = (uint64_t)src[i] << 32 | src[i];
  }
  if constexpr (line_vg(NQ, true) < line_vg(NQ, false))
    if (line_small<line_vg(NQ, false), line_vg(NQ, true)>(elems, sms))
      return launch_line_form<T, TS, NP, NQ, CPLX, BOX, kLineSmall>(c, lp, (elems + 1) / 2, sms, s);
  if constexpr (std::is_same<T, float>::value && NQ <= 9) {
    // wide form from one full tile of columns on; a unit's start (tables, first rows of X) costs about half a tile
    const int ntile = (ncg + S::VG - 1) / S::VG;
    if (ncg >= S::VG && (int64_t)prm.n_cells * ntile < (1LL << 30)) {
      lp.run = tiles_per_unit(prm.n_cells, ntile, (int64_t)WideShape<NP, NQ, CPLX, BOX>::MINB * sms, 0.5);
      return launch_line_form<T, TS, NP, NQ, CPLX, BOX, kLineWide>(
          c, lp, (int64_t)prm.n_cells * ((ntile + lp.run - 1) / lp.run), sms, s);
    }
  }
  return launch_line_form<T, TS, NP, NQ, CPLX, BOX, kLineFlat>(c, lp, (elems + S::VG - 1) / S::VG, sms, s);
}

}  // namespace feks
