// FP64-accurate Gram product C = Y^T Z of the Rayleigh-Ritz step (Algorithm 3)
// on the tensor cores, by exact integer slices (in the manner of Ozaki's
// error-free splitting of a matrix product into low-precision products).
//
// The product has a long contraction (the m DoF rows) and a small output
// (n x n, n = N_v): a dense contraction, but one that must be FP64-accurate.
// Rows are taken in chunks of R = 32.  For each chunk and each column of Y
// (and of Z), every value is written in fixed point relative to the column's
// largest exponent in the chunk (integer operations on its bit pattern) and
// cut into eight unsigned 7-bit slices c_0..c_7 (bits 63..8 of the aligned
// 64-bit significand; the sign goes with each slice):
//     y = 2^E sum_s (+-c_s) 2^(-7 s),  E = (largest biased exponent) - 1029.
// Each scaled slice (+-c_s) 2^(-7 s) is a BF16 number exactly, and a product
// of a Y slice and a Z slice is exact in FP32 (|c_s d_t| < 2^14).  The tensor
// cores add the products of a group of slice pairs in an FP32 accumulator.
// That accumulation was measured to behave like a truncating adder of about
// 21-22 significant bits (a first version's error matched such a model to
// within 10 %), so the grouping keeps every group whose loss could matter
// exact within 21 bits: the pairs with s + t = d for d = 0..4 each get an
// accumulator of their own (at most (d+1) x 32 x 127^2 < 2^21.3 in units of
// 2^(-7d); the d = 4 group may lose one bit, 2^(-49) of the result), and the
// pairs with s + t = 5..7 (at most 2^(-35) of the result) share a sixth.
// Pairs with s + t > 7 are dropped (below 2^(-56)).  The six accumulators of a
// 128 x 64 output tile take 384 of the 512 tensor-memory columns.
//
// After each chunk the tile is read back (tcgen05.ld), the six accumulators
// are combined in pairs of floats, scaled by 2^(E_i + E_j) and added to a
// running pair-of-floats sum per output in registers.  A CTA covers one
// 128 x 64 output tile and a group of rows; its FP64 partial goes to the same
// [group][n][n] workspace as the pair-of-floats Gram kernel, whose
// compensated, fixed-order reduction finishes the product.  Deterministic.
//
// Operand staging: a warp slices 8 columns of the tile (16 warps; Y's 128 columns, and
// warps 8..15 also Z's 64), a lane 8 of the chunk's 32 rows of one column: the column's
// largest exponent is two shuffles, and the lane's 8 values of a slice are one 16-byte
// row of the canonical K-major, no-swizzle layout (8 rows x 16 bytes per core matrix; core
// matrices 128 bytes apart along K, 512 bytes apart along M / N), a warp's rows 512
// contiguous bytes.  One thread issues the 72 MMAs of a chunk (36 slice pairs x 2 K-steps
// of 16), tcgen05.commit signals an mbarrier, all threads wait on it (bounded).
//
// What bounds it: instruction issue of the slicing (26 instructions a value) and of the
// readout (38 an output), not the MMAs.  So everything else is taken off the chain: two
// operand buffers, the next chunk sliced while this one's MMAs run and the one after
// loaded to registers meanwhile, one block barrier per chunk, and the readout split so that the
// warps that slice Z read fewer columns.  96 columns of 216000 rows: Gram 3.66 -> 0.64 ms, rotation
// 1.31 -> 0.72 ms.
#include <cuda_bf16.h>

#include <algorithm>

#include "fe_ks_internal.h"

namespace feks {
namespace tg {

constexpr int R = 32;                        // rows per chunk
constexpr int NS = 8;                        // 7-bit slices
constexpr int TILE = 128;                    // output tile rows (operand A rows, MMA M)
constexpr int TN = 64;                       // output tile columns (operand B rows, MMA N)
constexpr int NACC = 6;                      // accumulators: s + t = 0..4, and 5..7
constexpr int NT = 512;
constexpr uint32_t LBO = 128;                // K-direction core-matrix stride (bytes)
constexpr uint32_t SBO = 512;                // M/N-direction core-matrix stride (bytes)
constexpr int SLICE = TILE * R * 2;          // bytes of one A slice operand (8 KB)
constexpr int SLICE_B = TN * R * 2;          // bytes of one B slice operand (4 KB)
constexpr int OFF_A = 0;                     // within an operand buffer
constexpr int OFF_B = NS * SLICE;
constexpr int OPBUF = OFF_B + NS * SLICE_B;
constexpr int OFF_E = 2 * OPBUF;             // exponents of the operand rows, two buffers
constexpr int NE = TILE + TN;
constexpr int OFF_MBAR = OFF_E + 2 * NE * 4;
constexpr int OFF_TMEM = OFF_MBAR + 8;
constexpr int OFF_FLAG = OFF_TMEM + 4;
constexpr int BYTES = OFF_FLAG + 12;
constexpr uint32_t TMEM_COLS = 512;          // six 64-column FP32 accumulators (384 used)
constexpr long long kWaitIters = 1LL << 22;  // bound of an mbarrier wait (try_wait polls)

static_assert(TILE * R * 2 == SLICE && R % 16 == 0 && NACC * TN <= (int)TMEM_COLS, "chunk shape");

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((LBO >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((SBO >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version of the 5th-generation tensor core; no swizzle
  return d;
}

// kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, M = 128, N = 64
__host__ __device__ constexpr uint32_t idesc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TILE >> 4) << 24);
}

__device__ __forceinline__ void mma(uint32_t dt, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dt),
      "l"(a), "l"(b), "r"(idesc()), "r"(acc));
}

// 4 consecutive FP32 columns of this thread's tensor-memory lane
__device__ __forceinline__ void ld4(uint32_t ta, float (&v)[4]) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(ta));
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}

// bounded wait for phase `parity` of the mbarrier; returns false on expiry
__device__ __forceinline__ bool mbar_wait(uint32_t mb, uint32_t parity) {
  uint32_t done = 0;
  for (long long it = 0; it < kWaitIters && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mb), "r"(parity)
        : "memory");
  }
  return done != 0;
}

// hi + lo = a + b exactly (Knuth)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// Rows 8 g .. 8 g + 7 of a chunk of one operand row (zero from `count` on)
__device__ __forceinline__ void load_item(const double* __restrict__ src, int64_t stride, int count, int g,
                                          double (&v)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int r = 8 * g + q;
    v[q] = r < count ? src[(int64_t)r * stride] : 0.0;
  }
}

// Cut the lane's 8 values into the eight slice operands (row r8 of the 8-row group at `base`,
// K group g = lane / 8); returns the exponent E of the row's 32 values (four lanes).  A slice is
// seven bits of the aligned significand: put as they stand into the mantissa of a float 2^k, less
// 2^k, they are the slice's value exactly, and its BF16 number is that float's upper half.
__device__ __forceinline__ int slice_item(const double (&v)[8], uint32_t base, int slice_bytes, int r8, int g) {
  int emax = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int eb = (__double2hiint(v[q]) >> 20) & 0x7FF;
    emax = eb > emax ? eb : emax;
  }
  emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 8));
  emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 16));
  uint32_t w[NS][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t f[2][NS], sign = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(v[2 * q + h]);
      const int eb = (int)((b >> 52) & 0x7FFu), sh = emax - eb;
      unsigned long long al = 0ull;
      if (eb != 0 && sh < 64) al = (((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11) >> sh;
      const uint32_t hi = (uint32_t)(b >> 32);
      sign |= h ? (hi & 0x80000000u) : ((hi >> 16) & 0x8000u);
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const uint32_t x = s < 4 ? (uint32_t)(al >> 32) : (uint32_t)(al >> 4);   // four slices from bit 31 down
        const uint32_t field = ((s & 2) ? x : x >> 14) & ((s & 1) ? 0x7F0u : 0x3F800u);
        const uint32_t k = (uint32_t)(150 - ((s & 1) ? 4 : 11) - 7 * s) << 23;
        f[h][s] = __float_as_uint(__fsub_rn(__uint_as_float(field | k), __uint_as_float(k)));
      }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) w[s][q] = __byte_perm(f[0][s], f[1][s], 0x7632) ^ sign;
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const uint32_t a = base + s * slice_bytes + r8 * 16 + g * LBO;
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(a), "r"(w[s][0]), "r"(w[s][1]), "r"(w[s][2]),
                 "r"(w[s][3])
                 : "memory");
  }
  return emax - 1029;
}

// One thread: the chunk's 72 MMAs (pair (s, t) -> accumulator min(s + t, 5)), then commit.
__device__ __forceinline__ void issue_chunk(uint32_t s0, uint32_t tmem, uint32_t mbar) {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint64_t da = sdesc(s0 + OFF_A), db = sdesc(s0 + OFF_B);
#pragma unroll
  for (int d = 0; d < NS; ++d)
#pragma unroll
    for (int s = 0; s <= d; ++s)
#pragma unroll
      for (int ks = 0; ks < R / 16; ++ks) {
        const int t = d - s, g = d < NACC - 1 ? d : NACC - 1;
        const bool first = s == 0 && ks == 0 && d <= NACC - 1;   // the accumulator's first product of the chunk
        mma(tmem + (uint32_t)(g * TN), da + (uint64_t)((s * SLICE + ks * 2 * (int)LBO) >> 4),
            db + (uint64_t)((t * SLICE_B + ks * 2 * (int)LBO) >> 4), !first);
      }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar)
               : "memory");
}

// Columns of the tile read out by a warp: with two warps per lane quarter and half, warps 0..7
// take 20 columns each, warps 8..15 (which slice twice) 12.
constexpr int NB0 = 5, NB1 = 3;   // blocks of 4 columns
static_assert(2 * 4 * (NB0 + NB1) == TN, "readout split");

// Read this thread's outputs of the chunk (row orow of the tile, nb blocks of 4 columns from
// ocol0), combine the six accumulators in pairs of floats, scale by 2^(E_row + E_col) and add to the
// running pairs.  Every addition is error-free: the sum so far is a multiple of the units of the
// accumulators in it, so of the last place of the next one, and for such terms the three operations
// of Dekker's sum give the remainder whichever is larger.
__device__ __forceinline__ void accumulate_chunk(uint32_t tmem, int warp, int orow, int ocol0, int nb, const int* Es,
                                                 float (&acc_hi)[4 * NB0], float (&acc_lo)[4 * NB0], int* sflag) {
  const int Ei = Es[orow];
  const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)ocol0;
#pragma unroll
  for (int cb = 0; cb < NB0; ++cb) {
    if (cb >= nb) break;   // uniform in the warp
    float a[NACC][4];
#pragma unroll
    for (int g = 0; g < NACC; ++g) ld4(ta + (uint32_t)(g * TN + 4 * cb), a[g]);
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int jj = 4 * cb + j;
      const int E = Ei + Es[TILE + ocol0 + jj];
      float h = a[0][j], l = 0.f;
#pragma unroll
      for (int g = 1; g < NACC; ++g) {
        const float s = h + a[g][j];
        l += a[g][j] - (s - h);
        h = s;
      }
      if (E < -126 || E > 127) {
        if (h != 0.f || l != 0.f) *sflag = 1;
        continue;
      }
      const float sc = __uint_as_float((uint32_t)(E + 127) << 23);
      h *= sc;
      l *= sc;
      float s, e;   // running pair += (h, l)
      two_sum(acc_hi[jj], h, s, e);
      e += acc_lo[jj] + l;
      acc_hi[jj] = s + e;
      acc_lo[jj] = e - (acc_hi[jj] - s);
    }
  }
}

// MODE 0 (symmetric Gram C = Y^T Z): tile rows [128 blockIdx.y, +128), columns [64 blockIdx.x, +64),
//   skipped when every row index exceeds every column index; rows [rows blockIdx.z, +rows) of Y
//   and Z, chunks of 32 rows; partial -> part[blockIdx.z][n][n].
// MODE 1 (rotation X = Y E, Y [m][n], E [n][k]): column tile blockIdx.x of X, row tiles
//   blockIdx.y, blockIdx.y + gridDim.y, ... (persistent); chunks of 32 of the n contraction
//   indices; each row tile's result -> X.
// err[0]: a wait expired; err[1]: a chunk's scale 2^(E_i + E_j) left the FP32 range.
template <int MODE>
__global__ void __launch_bounds__(NT, 1) tc_slice_kernel(const double* __restrict__ Y, const double* __restrict__ Z,
                                                         double* __restrict__ out, int64_t m, int n, int k, int rows,
                                                         int* err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int ti = blockIdx.y, tj = blockIdx.x;
  if (MODE == 0 && ti * TILE > tj * TN + TN - 1) return;   // symmetric: a tile wholly below the diagonal
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
  int* Esm = reinterpret_cast<int*>(smem + OFF_E);
  const uint32_t mbar = s0 + OFF_MBAR;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + OFF_TMEM);
  int* sflag = reinterpret_cast<int*>(smem + OFF_FLAG);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mbar));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    *sflag = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(s0 + OFF_TMEM),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tslot;

  // slicing: warp w takes rows 8 w .. 8 w + 7 of operand A, warps 8..15 also rows of B
  const int r8 = lane & 7, g = lane >> 3;
  const int arow = 8 * warp + r8, brow = 8 * (warp - 8) + r8;
  const bool has_b = warp >= 8;
  const int orow = 32 * (warp & 3) + lane;     // readout: TMEM lane quarter
  const int nb = has_b ? NB1 : NB0;
  const int ocol0 = has_b ? 8 * NB0 + 4 * NB1 * ((warp - 8) >> 2) : 4 * NB0 * (warp >> 2);
  float acc_hi[4 * NB0], acc_lo[4 * NB0];
  bool failed = false;
  uint32_t phase = 0, failed_phase = 0;

  const int64_t ntile_r = MODE == 0 ? 1 : (m + TILE - 1) / TILE;
  for (int64_t tr = (MODE == 0 ? 0 : ti); tr < ntile_r && !failed; tr += (MODE == 0 ? 1 : gridDim.y)) {
#pragma unroll
    for (int j = 0; j < 4 * NB0; ++j) acc_hi[j] = acc_lo[j] = 0.f;
    int64_t c_begin, c_end;   // contraction range of this tile
    if (MODE == 0) {
      c_begin = (int64_t)blockIdx.z * rows;
      c_end = c_begin + rows < m ? c_begin + rows : m;
    } else {
      c_begin = 0;
      c_end = n;
    }
    const int nch = (int)((c_end - c_begin + R - 1) / R);
    double va[8], vb[8];
    auto load = [&](int ch) {
      const int64_t c0 = c_begin + (int64_t)ch * R;
      const int cnt = (int)(c_end - c0 < R ? c_end - c0 : R);
      if (MODE == 0) {
        const int col = ti * TILE + arow;
        load_item(Y + c0 * n + col, n, col < n ? cnt : 0, g, va);
      } else {
        const int64_t row = tr * TILE + arow;
        load_item(Y + row * n + c0, 1, row < m ? cnt : 0, g, va);
      }
      if (has_b) {
        const int col = tj * TN + brow;
        load_item(Z + c0 * k + col, k, col < k ? cnt : 0, g, vb);   // MODE 0: k = n
      }
    };
    auto slice = [&](int ch) {
      const uint32_t op = s0 + (ch & 1) * OPBUF;
      int* Es = Esm + (ch & 1) * NE;
      const int ea = slice_item(va, op + OFF_A + warp * SBO, SLICE, r8, g);
      if (g == 0) Es[arow] = ea;
      if (has_b) {
        const int eb = slice_item(vb, op + OFF_B + (warp - 8) * SBO, SLICE_B, r8, g);
        if (g == 0) Es[TILE + brow] = eb;
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    };
    load(0);
    slice(0);
    if (nch > 1) load(1);
    __syncthreads();
    for (int ch = 0; ch < nch; ++ch) {
      // this chunk's MMAs run beside the next one's slicing and the loads of the one after; the buffer
      // being written was last read by the MMAs of chunk ch - 1, waited for below
      if (tid == 0) issue_chunk(s0 + (ch & 1) * OPBUF, tmem, mbar);
      __syncwarp();
      if (ch + 1 < nch) slice(ch + 1);
      if (ch + 2 < nch) load(ch + 2);
      const bool ok = mbar_wait(mbar, phase);
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      __syncwarp();
      accumulate_chunk(tmem, warp, orow, ocol0, nb, Esm + (ch & 1) * NE, acc_hi, acc_lo, sflag);
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      if (__syncthreads_or(!ok)) {   // the next chunk overwrites the accumulators
        failed = true;
        failed_phase = phase;
        break;
      }
      phase ^= 1u;
    }
    if (failed) break;
    if (MODE == 0) {
      double* o = out + (int64_t)blockIdx.z * n * n;
      const int i = ti * TILE + orow;
      if (i < n)
#pragma unroll
        for (int jj = 0; jj < 4 * NB0; ++jj) {
          const int j = tj * TN + ocol0 + jj;
          if (jj < 4 * nb && j < n) o[(int64_t)i * n + j] = (double)acc_hi[jj] + (double)acc_lo[jj];
        }
    } else {
      const int64_t row = tr * TILE + orow;
      if (row < m)
#pragma unroll
        for (int jj = 0; jj < 4 * NB0; ++jj) {
          const int j = tj * TN + ocol0 + jj;
          if (jj < 4 * nb && j < k) out[row * k + j] = (double)acc_hi[jj] + (double)acc_lo[jj];
        }
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (failed) atomicExch(err, 1);
    if (*sflag) atomicExch(err + 1, 1);
  }
  if (failed && tid == 0) {
    // give MMAs still in flight a last bounded chance to drain before the tensor memory is released
    (void)mbar_wait(mbar, failed_phase);
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
}

// shared-memory opt-in of a kernel mode, once per device
template <int MODE>
fe_ks_status prepare() {
  static bool done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!done[dev & 63]) {
    cudaError_t e = cudaFuncSetAttribute(tc_slice_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, BYTES);
    if (e != cudaSuccess) return fail(FE_KS_ERR_CUDA, std::string("tensor-core slice kernel attribute: ") + cudaGetErrorString(e));
    done[dev & 63] = true;
  }
  return FE_KS_OK;
}

}  // namespace tg
}  // namespace feks

using namespace feks;

extern "C" {

// Row groups of the Gram product: as many as fill the device once (one CTA per SM: the
// accumulators take the tensor memory), or a multiple of that once a group would exceed
// kGramChunkRows; at least kGramMinRows rows each.  96 columns of 216000 rows took
// 3.66 ms in groups of 8192 rows (54 CTAs on 152 SMs).
static int64_t gram_groups(int64_t m, int n) {
  constexpr int64_t kGramMinRows = 256;
  int64_t tiles = 0;
  for (int ti = 0; ti * tg::TILE < n; ++ti)
    for (int tj = 0; tj * tg::TN < n; ++tj) tiles += ti * tg::TILE <= tj * tg::TN + tg::TN - 1;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 152;
  int64_t g = 0;
  for (int64_t w = 1; g * kGramChunkRows < m; ++w) g = std::max<int64_t>(w, w * sms / tiles);
  return std::min(g, std::max((m + kGramMinRows - 1) / kGramMinRows, (m + kGramChunkRows - 1) / kGramChunkRows));
}

fe_ks_status fe_ks_gram_tc_workspace(int64_t m, int n, size_t* bytes) {
  set_error("");
  if (!bytes || m < 1 || n < 1) return fail(FE_KS_ERR_ARG, "bad sizes");
  size_t b = 0;
  fe_ks_status st = fe_ks_gram_ff_workspace(m, n, n, &b);
  if (st != FE_KS_OK) return st;
  b = std::max(b, (size_t)gram_groups(m, n) * n * n * sizeof(double));
  *bytes = b + 256;   // two status words (first 256 bytes), then the partials
  return FE_KS_OK;
}

fe_ks_status fe_ks_gram_tc_sym(const double* Y, const double* Z, double* C, int64_t m, int n, void* work,
                               size_t work_bytes, void* cuda_stream) {
  set_error("");
  if (!Y || !Z || !C || !work) return fail(FE_KS_ERR_ARG, "NULL argument");
  size_t need = 0;   // the least: groups of kGramChunkRows rows
  if (m < 1 || n < 1) return fail(FE_KS_ERR_ARG, "bad sizes");
  fe_ks_status st = fe_ks_gram_ff_workspace(m, n, n, &need);
  if (st != FE_KS_OK) return st;
  need += 256;
  if (work_bytes < need) return fail(FE_KS_ERR_ARG, "workspace too small");
  if (((uintptr_t)work & 255) || ((uintptr_t)Y & 7) || ((uintptr_t)Z & 7)) return fail(FE_KS_ERR_ARG, "misaligned argument");
  const int64_t fit = (int64_t)((work_bytes - 256) / ((size_t)n * n * sizeof(double)));
  const int64_t groups = std::min(gram_groups(m, n), fit);
  const int rows = (int)(((m + groups - 1) / groups + tg::R - 1) / tg::R * tg::R);
  const int64_t nch = (m + rows - 1) / rows;
  if (nch > 65535 || n > 4096) return fail(FE_KS_ERR_ARG, "sizes too large for the tensor-core Gram kernel");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  int* flags = static_cast<int*>(work);
  double* part = reinterpret_cast<double*>(static_cast<char*>(work) + 256);
  fe_ks_status ast = tg::prepare<0>();
  if (ast != FE_KS_OK) return ast;
  if (cudaMemsetAsync(flags, 0, 2 * sizeof(int), s) != cudaSuccess) return fail(FE_KS_ERR_CUDA, "cudaMemsetAsync");
  dim3 grid((unsigned)((n + tg::TN - 1) / tg::TN), (unsigned)((n + tg::TILE - 1) / tg::TILE), (unsigned)nch);
  tg::tc_slice_kernel<0><<<grid, tg::NT, tg::BYTES, s>>>(Y, Z, part, m, n, n, rows, flags);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_gram_reduce(part, C, (int)nch, n, n, 1, s);
  if (e != cudaSuccess) return fail(FE_KS_ERR_CUDA, std::string("tensor-core Gram kernels: ") + cudaGetErrorString(e));
  return FE_KS_OK;
}

fe_ks_status fe_ks_rotate_tc(const double* Y, const double* E, double* X, int64_t m, int n, int k, int* flags,
                             void* cuda_stream) {
  set_error("");
  if (!Y || !E || !X || !flags) return fail(FE_KS_ERR_ARG, "NULL argument");
  if (m < 1 || n < 1 || k < 1 || n > 4096 || k > 4096) return fail(FE_KS_ERR_ARG, "bad sizes");
  if (((uintptr_t)Y & 7) || ((uintptr_t)E & 7) || ((uintptr_t)X & 7) || ((uintptr_t)flags & 3))
    return fail(FE_KS_ERR_ARG, "misaligned argument");
  fe_ks_status ast = tg::prepare<1>();
  if (ast != FE_KS_OK) return ast;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemsetAsync(flags, 0, 2 * sizeof(int), s) != cudaSuccess) return fail(FE_KS_ERR_CUDA, "cudaMemsetAsync");
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int kt = (k + tg::TN - 1) / tg::TN;
  const int64_t rt = (m + tg::TILE - 1) / tg::TILE;
  const int64_t want = ((int64_t)(sms > 0 ? sms : 152) + kt - 1) / kt;   // about one CTA per SM, persistent
  const unsigned gy = (unsigned)(rt < want ? rt : want);
  tg::tc_slice_kernel<1><<<dim3((unsigned)kt, gy), tg::NT, tg::BYTES, s>>>(Y, E, X, m, n, k, 0, flags);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(FE_KS_ERR_CUDA, std::string("tensor-core rotation kernel: ") + cudaGetErrorString(e));
  return FE_KS_OK;
}

fe_ks_status fe_ks_gram_tc_status(const void* work, int* status) {
  set_error("");
  if (!work || !status) return fail(FE_KS_ERR_ARG, "bad arguments");
  int f[2] = {0, 0};
  const int* flags = static_cast<const int*>(work);
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(f, flags, sizeof(f), cudaMemcpyDeviceToHost) != cudaSuccess)
    return fail(FE_KS_ERR_CUDA, "reading the Gram status failed");
  *status = (f[0] ? 1 : 0) | (f[1] ? 2 : 0);
  return FE_KS_OK;
}

}  // extern "C"
