// Default cell kernel of the FP64-accurate pair-of-floats precision.
//
// Same slots, lines and assembly as fe_ks_line.cuh.  A contraction of one line costs
// ten times the instructions of an FP32 one here, so what matters is not the
// shared-memory traffic but that the instructions stay in the cache: every 1D
// operator is written once and looped over the three directions with run-time
// strides (four line bodies instead of twelve), the quadrature-point step is a rolled loop
// over a line's points, and the z derivative has a shared tile of its own.
//   N_z, N_y, N_x on A;  D~_z, D~_y, D~_x: A -> B[2], B[1], B[0];  point step;
//   A += D~_z^T B[2], D~_y^T B[1], D~_x^T B[0];  N_x^T, N_y^T, N_z^T on A; assembly.
#pragma once
#include "fe_ks_line.cuh"

namespace feks {

// y = M x (see eo_apply) in the pair arithmetic of fe_ks_ff.cuh; every y[o] goes to
// put(o, y) as soon as it is formed, so that only the butterflies stay in registers
template <int NI, int NO, int S, class Put>
__device__ __forceinline__ void eo_apply_ff(const ff2* x, const EOMat<ff2>& m, Put put) {
  constexpr int HI = NI / 2, HO = NO / 2;
  ff2 xe[HI], xo[HI];
#pragma unroll
  for (int i = 0; i < HI; ++i) {
    xe[i] = ff_add(x[i], x[NI - 1 - i]);
    xo[i] = ff_add(x[i], -x[NI - 1 - i]);
  }
#pragma unroll
  for (int o = 0; o < HO; ++o) {
    ff2 ye = ff_mul(m.E[o][0], xe[0]);
#pragma unroll
    for (int i = 1; i < HI; ++i) ye = ff_fma(m.E[o][i], xe[i], ye);
    if (NI % 2) ye = ff_fma(m.E[o][HI], x[HI], ye);
    ff2 yo = ff_mul(m.O[o][0], xo[0]);
#pragma unroll
    for (int i = 1; i < HI; ++i) yo = ff_fma(m.O[o][i], xo[i], yo);
    put(o, ff_add(ye, yo));
    put(NO - 1 - o, S > 0 ? ff_add(ye, -yo) : ff_add(yo, -ye));
  }
  if (NO % 2) {
    ff2 ym = ff_mul(m.MID[0], S > 0 ? xe[0] : xo[0]);
#pragma unroll
    for (int i = 1; i < HI; ++i) ym = ff_fma(m.MID[i], S > 0 ? xe[i] : xo[i], ym);
    if (S > 0 && NI % 2) ym = ff_fma(m.MID[HI], x[HI], ym);
    put(HO, ym);
  }
}

// Four tiles per block; VG, NT, MINB and SMALL as in LineShape.  Measured at 10^3 cells, 64 columns, for
// two-element tiles / these: p = 8 3576 / 2820 us, p = 7 1914 / 1590, p = 6 1472 / 1164, p = 5 963 / 662,
// p = 4 420 / 376.
constexpr int line_ff_vg(int nq, bool small) { return small ? 2 : nq >= 10 ? 2 : nq >= 8 ? 4 : nq >= 5 ? 8 : 16; }
constexpr int line_ff_minb(int nq, bool small, int nt) {
  return small ? (768 / nt < 16 ? 768 / nt : 16)
               : nq >= 11 ? 2 : nq == 10 ? 3 : nq == 9 ? 2 : nq == 8 ? 3 : nq == 7 ? 2 : nq == 6 ? 3 : nq == 5 ? 4 : nq == 4 ? 3 : nq == 3 ? 6 : 12;
}
template <int NQ, bool SMALL = false>
struct LineShapeFF {
  static constexpr int VG = line_ff_vg(NQ, SMALL);
  static constexpr int NT = (NQ * NQ * VG + 31) / 32 * 32;
  static constexpr int MINB = line_ff_minb(NQ, SMALL, NT);
  static constexpr int PY = NQ | 1;
  static constexpr int SX = VG, SY = PY * VG, SZ = NQ * SY, BUF = NQ * SZ;
  static constexpr size_t bytes = 4 * (size_t)BUF * 8;
};

// line_small by the pairs' own widths.  At n_q = 7 a full tile has eight elements and two-element tiles
// must save a quarter (p = 6, small / full: 512 slots 24.7 / 34.9 us, 2496 64.8 / 69.7; where they save
// less: 3000 76 / 70, 5145 125 / 111).
template <int NQ>
bool line_ff_small(int64_t slots, int sms) {
  return line_small<line_ff_vg(NQ, false), line_ff_vg(NQ, true), NQ == 7 ? 6 : 7>(slots, sms);
}

template <int NP, int NQ, bool CPLX, bool SMALL>
__global__ void __launch_bounds__(LineShapeFF<NQ, SMALL>::NT, LineShapeFF<NQ, SMALL>::MINB)
    fe_line_ff_kernel(const __grid_constant__ LocalParams<ff2, double> p, int per_sm) {
  using S = LineShapeFF<NQ, SMALL>;
  using E = Elem<ff2, double>;
  constexpr int VG = S::VG, SX = S::SX, SY = S::SY, SZ = S::SZ, NQ2 = NQ * NQ, NQ3 = NQ * NQ2, NP2 = NP * NP;
  constexpr int NP3 = NP * NP2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int v = threadIdx.x % VG, ln = threadIdx.x / VG;
  ff2* const A = reinterpret_cast<ff2*>(smem_raw) + v;
  ff2* const B = A + S::BUF;   // B[ax] at B + ax BUF
  const int64_t nslots = (int64_t)p.n_cells * p.ncols;
  const int64_t ntiles = (nslots + VG - 1) / VG;
  const bool gauss_line = ln < NQ2;
  const unsigned gmask = CPLX ? __ballot_sync(0xffffffffu, gauss_line) : 0u;
  // In full rounds the blocks that share a multiprocessor (b, b + sms, ...) take neighbouring tiles, so
  // that its L1 serves a cell's coefficients to them (8^3 cells, p = 8, 64 columns: 1770 -> 1697 us);
  // the last round spreads over the multiprocessors.
  const int sms = gridDim.x / per_sm, near = (int)(blockIdx.x % sms) * per_sm + (int)(blockIdx.x / sms);
  const int64_t full = ntiles / gridDim.x * gridDim.x;
  for (int64_t r = 0; r < ntiles; r += gridDim.x) {
    const int64_t t = r + (r < full ? near : (int)blockIdx.x);
    if (t >= ntiles) break;
    // an idle lane repeats a slot of its own re/im parity and stores nothing
    const int64_t slot = t * VG + v;
    const bool act = slot < nslots;
    const int ci = act ? (int)(slot / p.ncols) : p.n_cells - 1;
    const int col = act ? (int)(slot - (int64_t)ci * p.ncols) : CPLX ? (int)(slot & 1) : 0;
    const int e = p.cells ? p.cells[ci] : ci;
    // N along z (from the gathered rows of X), y, x
#pragma unroll 1
    for (int ax = 2; ax >= 0; --ax) {
      const int lines = ax == 2 ? NP2 : ax == 1 ? NP * NQ : NQ2, n0 = ax == 0 ? NQ : NP;
      const int sp = ax == 2 ? SZ : ax == 1 ? SY : SX;
      ff2* a = A + (ln % n0) * (ax == 0 ? SY : SX) + (ln / n0) * (ax == 2 ? SY : SZ);
      if (ln < lines) {
        ff2 x[NP];
        if (ax == 2) {
          const int* __restrict__ dofs = p.cell_dofs + (int64_t)e * NP3 + ln;
#pragma unroll
          for (int k = 0; k < NP; ++k) {
            const int d = dofs[k * NP2];
            x[k] = E::load(p.X + (int64_t)d * p.ld + col, true, true);
            if (p.dscale) x[k] = p.dscale[d] * x[k];
          }
        } else {
#pragma unroll
          for (int k = 0; k < NP; ++k) x[k] = a[k * sp];
        }
        eo_apply_ff<NP, NQ, 1>(x, p.tab.N, [&](int q, ff2 y) { a[q * sp] = y; });
      }
      __syncthreads();
    }
    // D~ along z, y, x
    if (gauss_line) {
#pragma unroll 1
      for (int ax = 2; ax >= 0; --ax) {
        const int sp = ax == 2 ? SZ : ax == 1 ? SY : SX;
        const int o = (ln % NQ) * (ax == 0 ? SY : SX) + (ln / NQ) * (ax == 2 ? SY : SZ);
        ff2 x[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) x[q] = A[o + q * sp];
        ff2* b = B + ax * S::BUF + o;
        eo_apply_ff<NQ, NQ, -1>(x, p.tab.D, [&](int q, ff2 y) { b[q * sp] = y; });
      }
    }
    __syncthreads();
    // Z = V^L Y0 + V^G.grad - i V^K.grad, W_s = sum_d G_sd grad_d + V^G_s Y0, one z line per thread
    if (gauss_line) {
      // the next point's coefficients load while this one's are used
      constexpr int NCF = CPLX ? kCoefCplx : kCoefReal;
      const ff2* __restrict__ cf = p.coef + (int64_t)e * p.ncoef * NQ3 + ln;
      ff2 c[NCF];
#pragma unroll
      for (int k = 0; k < NCF; ++k) c[k] = cf[k * NQ3];
      int s = (ln % NQ) * SX + (ln / NQ) * SY;
#pragma unroll 1
      for (int q = 0; q < NQ; ++q, s += SZ) {
        ff2 cn[NCF];
        cf += q + 1 < NQ ? NQ2 : 0;
#pragma unroll
        for (int k = 0; k < NCF; ++k) cn[k] = cf[k * NQ3];
        const ff2 uu = A[s], gx = B[s], gy = B[S::BUF + s], gz = B[2 * S::BUF + s];
        ff2 z = ff_mul(c[6], uu);
        ff2 w0 = ff_fma(c[0], gx, ff_fma(c[1], gy, ff_mul(c[2], gz)));
        ff2 w1 = ff_fma(c[1], gx, ff_fma(c[3], gy, ff_mul(c[4], gz)));
        ff2 w2 = ff_fma(c[2], gx, ff_fma(c[4], gy, ff_mul(c[5], gz)));
        if (p.gga) {
          z = ff_fma(c[7], gx, ff_fma(c[8], gy, ff_fma(c[9], gz, z)));
          w0 = ff_fma(c[7], uu, w0);
          w1 = ff_fma(c[8], uu, w1);
          w2 = ff_fma(c[9], uu, w2);
        }
        if constexpr (CPLX) {
          const ff2 kk = ff_fma(c[10], gx, ff_fma(c[11], gy, ff_mul(c[12], gz)));
          z = ff_add(z, E::minus_i(kk, v, gmask));
        }
        A[s] = z;
        B[s] = w0;
        B[S::BUF + s] = w1;
        B[2 * S::BUF + s] = w2;
#pragma unroll
        for (int k = 0; k < NCF; ++k) c[k] = cn[k];
      }
    }
    __syncthreads();
    // A += D~^T B[ax] along z, y, x
#pragma unroll 1
    for (int ax = 2; ax >= 0; --ax) {
      if (gauss_line) {
        const int sp = ax == 2 ? SZ : ax == 1 ? SY : SX;
        const int o = (ln % NQ) * (ax == 0 ? SY : SX) + (ln / NQ) * (ax == 2 ? SY : SZ);
        const ff2* b = B + ax * S::BUF + o;
        ff2 x[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) x[q] = b[q * sp];
        eo_apply_ff<NQ, NQ, -1>(x, p.tab.Dt,
                                [&](int q, ff2 y) { A[o + q * sp] = ff_add(A[o + q * sp], y); });
      }
      __syncthreads();
    }
    // N^T along x, y, z; the last lines are a node's z lines: expansion and assembly
#pragma unroll 1
    for (int ax = 0; ax < 3; ++ax) {
      const int lines = ax == 2 ? NP2 : ax == 1 ? NP * NQ : NQ2, n0 = ax == 0 ? NQ : NP;
      const int sp = ax == 2 ? SZ : ax == 1 ? SY : SX;
      ff2* a = A + (ln % n0) * (ax == 0 ? SY : SX) + (ln / n0) * (ax == 2 ? SY : SZ);
      if (ln < lines) {
        ff2 x[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) x[q] = a[q * sp];
        // the last lines, too, go through the tile (own line only): one copy of the operator's code
        eo_apply_ff<NQ, NP, 1>(x, p.tab.Nt, [&](int k, ff2 y) { a[k * sp] = y; });
        if (ax == 2 && act) {
          ff2 y[NP];
#pragma unroll
          for (int k = 0; k < NP; ++k) y[k] = a[k * sp];
          if (p.cell_pair_ptr) {
            const int pb = p.cell_pair_ptr[e], pe = p.cell_pair_ptr[e + 1];
            for (int pi = pb; pi < pe; ++pi) {
              const int pr = p.cell_pairs[pi];
              const double* Qa = p.Q + (int64_t)p.pair_atom[pr] * p.n_proj * p.ld;
              const ff2* __restrict__ Fp = p.F + ((int64_t)pr * p.n_proj * NP3 + ln) * (CPLX ? 2 : 1);
#pragma unroll 1
              for (int b = 0; b < p.n_proj; ++b) {
                const ff2 q = E::load(Qa + (int64_t)b * p.ld + col, true, true);
                const ff2* __restrict__ Fb = Fp + (int64_t)b * NP3 * (CPLX ? 2 : 1);
                if constexpr (!CPLX) {
#pragma unroll
                  for (int k = 0; k < NP; ++k) y[k] = ff_fma(Fb[k * NP2], q, y[k]);
                } else {
                  // (fr + i fi)(qr + i qi): re: fr qr - fi qi, im: fr qi + fi qr
                  const ff2 qp = E::load(Qa + (int64_t)b * p.ld + (col ^ 1), true, true);
                  const ff2 iq = (col & 1) ? qp : -qp;
#pragma unroll
                  for (int k = 0; k < NP; ++k)
                    y[k] = ff_fma(Fb[k * NP2 * 2], q, ff_fma(Fb[k * NP2 * 2 + 1], iq, y[k]));
                }
              }
            }
          }
          const int* __restrict__ dofs = p.cell_dofs + (int64_t)e * NP3 + ln;
          const int* __restrict__ dst = p.dst ? p.dst + (int64_t)e * NP3 + ln : nullptr;
#pragma unroll
          for (int k = 0; k < NP; ++k) {
            ff2 val = p.alpha * y[k];
            if (p.dscale) val = p.dscale[dofs[k * NP2]] * val;
            if (dst) {   // one launch for all cells: rows of one cell straight to Y, shared rows to their slots
              const int d = dst[k * NP2];
              if (d >= 0)
                E::store(p.Y + (int64_t)d * p.ld + col, val, true, true, p.accum);
              else
                E::store(p.W + (int64_t)(~d) * p.ld + col, val, true, true, false);
            } else {     // one colour: no two cells of the launch share a row of Y
              E::add(p.Y + (int64_t)dofs[k * NP2] * p.ld + col, val, true, true);
            }
          }
        }
      }
      if (ax < 2) __syncthreads();
    }
  }
}

template <int NP, int NQ, bool CPLX, bool SMALL>
cudaError_t launch_line_ff_form(const Ctx& c, const LocalParams<ff2, double>& prm, int sms, cudaStream_t s) {
  using S = LineShapeFF<NQ, SMALL>;
  static bool attr_done[64] = {};
  const int dev = c.device & 63;
  auto k = fe_line_ff_kernel<NP, NQ, CPLX, SMALL>;
  if (!attr_done[dev]) {
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::bytes);
    if (err != cudaSuccess) return err;
    attr_done[dev] = true;
  }
  const int64_t ntiles = ((int64_t)prm.n_cells * prm.ncols + S::VG - 1) / S::VG, slots = (int64_t)S::MINB * sms;
  k<<<(int)(ntiles < slots ? ntiles : slots), S::NT, S::bytes, s>>>(prm, ntiles < slots ? 1 : S::MINB);
  return cudaGetLastError();
}

template <int NP, int NQ, bool CPLX>
cudaError_t launch_line_ff_t(const Ctx& c, const LocalParams<ff2, double>& prm, cudaStream_t s) {
  const int sms = c.sms > 0 ? c.sms : 152;
  if (prm.n_cells == 0) return cudaSuccess;
  if constexpr (line_ff_vg(NQ, false) > 2)
    if (line_ff_small<NQ>((int64_t)prm.n_cells * prm.ncols, sms)) return launch_line_ff_form<NP, NQ, CPLX, true>(c, prm, sms, s);
  return launch_line_ff_form<NP, NQ, CPLX, false>(c, prm, sms, s);
}

}  // namespace feks
