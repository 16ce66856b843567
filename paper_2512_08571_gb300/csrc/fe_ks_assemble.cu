// One-launch assembly Q^T (Algorithm 1): sums of the shared rows.
//
// A cell kernel that runs all cells in one launch stores the rows that only one
// cell meets straight to Y and every other cell value to a slot of W of its own;
// the slots of a DoF are consecutive, in the order of the cells' colours.  The sum below then
// reads each slot once, adds a DoF's slots in that order (deterministic, no atomics, the bits
// of the colour-by-colour scatter) and writes its row of Y once.  Bound by the L2: 8^3 cells at p = 6
// with 48 FP32 columns have 21 MB in slots, summed in 7.3 us; it replaces a zero-fill of Y and a
// launch, with its tail, for all but one of the colours.
#include <algorithm>

#include "fe_ks_internal.h"

namespace feks {

// V columns per thread (V = 4 or 2 doubles / floats as one vector, or 1)
template <typename T, typename TV, int V>
__global__ void __launch_bounds__(256) fe_assemble_kernel(const T* __restrict__ W, T* __restrict__ Y, int64_t ld,
                                                          const int* __restrict__ dof, const int* __restrict__ ptr,
                                                          int64_t total, int groups, int accum) {
  for (int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x; i < total; i += (int64_t)gridDim.x * 256) {
    // 32-bit division wherever the index fits
    const int64_t s = i <= 0xFFFFFFFFll ? (int64_t)((uint32_t)i / (uint32_t)groups) : i / groups;
    const int64_t col = (i - s * groups) * V;
    const int b = ptr[s], e = ptr[s + 1];
    T* y = Y + (int64_t)dof[s] * ld + col;
    TV v = *reinterpret_cast<const TV*>(accum ? y : W + (int64_t)b * ld + col);
    T* a = reinterpret_cast<T*>(&v);
    for (int k = accum ? b : b + 1; k < e; ++k) {
      const TV w = *reinterpret_cast<const TV*>(W + (int64_t)k * ld + col);
      const T* wv = reinterpret_cast<const T*>(&w);
#pragma unroll
      for (int u = 0; u < V; ++u) a[u] += wv[u];
    }
    *reinterpret_cast<TV*>(y) = v;
  }
}

template <typename T, typename TV, int V>
static cudaError_t assemble_v(const Ctx& c, T* Y, int64_t ncols, int accum, cudaStream_t s) {
  const int64_t total = c.n_shared * (ncols / V);
  const int blocks = (int)std::min<int64_t>((total + 255) / 256, (int64_t)std::max(c.sms, 1) * 32);
  fe_assemble_kernel<T, TV, V><<<blocks, 256, 0, s>>>(asm_slots<T>(c), Y, ncols, c.asm_dof, c.asm_ptr,
                                                     total, (int)(ncols / V), accum);
  return cudaGetLastError();
}

template <>
cudaError_t launch_assemble<float>(const Ctx& c, float* Y, int64_t ncols, int accum, cudaStream_t s) {
  if (c.n_shared == 0) return cudaSuccess;
  if (ncols % 4 == 0 && (uintptr_t)Y % 16 == 0) return assemble_v<float, float4, 4>(c, Y, ncols, accum, s);
  if (ncols % 2 == 0 && (uintptr_t)Y % 8 == 0) return assemble_v<float, float2, 2>(c, Y, ncols, accum, s);
  return assemble_v<float, float, 1>(c, Y, ncols, accum, s);
}
template <>
cudaError_t launch_assemble<double>(const Ctx& c, double* Y, int64_t ncols, int accum, cudaStream_t s) {
  if (c.n_shared == 0) return cudaSuccess;
  if (ncols % 2 == 0 && (uintptr_t)Y % 16 == 0) return assemble_v<double, double2, 2>(c, Y, ncols, accum, s);
  return assemble_v<double, double, 1>(c, Y, ncols, accum, s);
}

}  // namespace feks
