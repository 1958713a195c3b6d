#pragma once
#include "camp_internal.h"
namespace camp {
// the automatic choice (at most 3 rows per lane on 8, 16 or 32 lanes, and 4 or
// 5 on 32) runs kernels with the lane count fixed at compile time
template <int E>
const void *mixed_kernel_of(int Lc) {
  if constexpr (E >= 2 && E <= 5)
    if (Lc == 32) return (const void *)mixed_refine_kernel<E, 32>;
  if constexpr (E >= 2 && E <= 3) {
    if (Lc == 16) return (const void *)mixed_refine_kernel<E, 16>;
    if (Lc == 8) return (const void *)mixed_refine_kernel<E, 8>;
  }
  return (const void *)mixed_refine_kernel<E, 0>;
}
}  // namespace camp
#define CAMP_MIXED_DEFINE(E)                                                              \
  cudaError_t launch_mixed_##E(const MixedArgs &a, int wpb, int grid, size_t smem,        \
                               cudaStream_t st) {                                         \
    const void *fn = mixed_kernel_of<E>(a.Lc);                                            \
    cudaError_t e = ensure_max_smem(fn);                                                  \
    if (e != cudaSuccess) return e;                                                       \
    void *args[] = {(void *)&a};                                                          \
    return a.ord_ws                                                                       \
               ? cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(wpb * 32), args, smem, st) \
               : cudaLaunchKernel(fn, dim3(grid), dim3(wpb * 32), args, smem, st);        \
  }                                                                                       \
  cudaError_t occ_mixed_##E(int Lc, int wpb, size_t smem, int *blocks) {                  \
    const void *fn = mixed_kernel_of<E>(Lc);                                              \
    cudaError_t e = ensure_max_smem(fn);                                                  \
    if (e != cudaSuccess) return e;                                                       \
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, fn, wpb * 32, smem);     \
  }
