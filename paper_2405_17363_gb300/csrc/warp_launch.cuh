// Per-E kernel tables, launch and occupancy entry points of the warp-packed
// kernels (plain solve, fused assembly, Newton), defined in the instantiation
// units and dispatched from solver.cu.
//
// The arrangements the automatic choice makes for 21..160 rows (3 to 5 rows
// per lane on 8, 16 or 32 lanes) run kernels with the lane count fixed at
// compile time: constant strides fold into the shared-memory addressing.  A
// launch that orders its cells itself (a.ord_ws set) is cooperative: its grid
// barrier needs every CTA resident.
#pragma once
#include "camp_internal.h"

namespace camp {
template <int E>
constexpr bool kFixedLanes = E >= 3 && E <= kRegVecMaxE;

template <int E>
const void *warp_kernel_of(int Lc, int tk) {
  if constexpr (E <= kRegVecMaxE) {
    if (Lc == 16 && tk == kTicketsOne) return (const void *)warp_bicgstab_kernel<E, 16, kTicketsOne>;
    if (Lc == 16 && tk == kTicketsBoth) return (const void *)warp_bicgstab_kernel<E, 16, kTicketsBoth>;
  }
  if constexpr (kFixedLanes<E>) {
    if (Lc == 8) return (const void *)warp_bicgstab_kernel<E, 8, kTicketsPack>;
    if (Lc == 16) return (const void *)warp_bicgstab_kernel<E, 16, kTicketsPack>;
    if (Lc == 32) return (const void *)warp_bicgstab_kernel<E, 32, kTicketsPack>;
  }
  return (const void *)warp_bicgstab_kernel<E, 0, kTicketsPack>;
}
template <int E>
const void *assemble_kernel_of(int Lc, int) {
  if constexpr (kFixedLanes<E>) {
    if (Lc == 8) return (const void *)assemble_bicgstab_kernel<E, 8>;
    if (Lc == 16) return (const void *)assemble_bicgstab_kernel<E, 16>;
    if (Lc == 32) return (const void *)assemble_bicgstab_kernel<E, 32>;
  }
  return (const void *)assemble_bicgstab_kernel<E, 0>;
}
template <int E>
const void *newton_kernel_of(int Lc, int) {
  if constexpr (kFixedLanes<E>) {
    if (Lc == 8) return (const void *)newton_bicgstab_kernel<E, 8>;
    if (Lc == 16) return (const void *)newton_bicgstab_kernel<E, 16>;
    if (Lc == 32) return (const void *)newton_bicgstab_kernel<E, 32>;
  }
  return (const void *)newton_bicgstab_kernel<E, 0>;
}

inline cudaError_t launch_kernel(const void *fn, const WarpArgs &a, int wpb, int grid, size_t smem,
                                 cudaStream_t st) {
  cudaError_t e = ensure_max_smem(fn);
  if (e != cudaSuccess) return e;
  void *args[] = {(void *)&a};
  return a.ord_ws ? cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(wpb * 32), args, smem, st)
                  : cudaLaunchKernel(fn, dim3(grid), dim3(wpb * 32), args, smem, st);
}
inline cudaError_t kernel_occupancy(const void *fn, int wpb, size_t smem, int *blocks) {
  cudaError_t e = ensure_max_smem(fn);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, fn, wpb * 32, smem);
}
}  // namespace camp

// launch_<name>_<E> and occ_<name>_<E> of the kernels <name>_kernel_of<E>
#define CAMP_KERNEL_DEFINE(name, E)                                                        \
  cudaError_t launch_##name##_##E(const WarpArgs &a, int wpb, int grid, size_t smem,       \
                                  cudaStream_t st) {                                       \
    return launch_kernel(name##_kernel_of<E>(a.Lc, tickets_of(a)), a, wpb, grid, smem, st); \
  }                                                                                        \
  cudaError_t occ_##name##_##E(int Lc, int tk, int wpb, size_t smem, int *blocks) {        \
    return kernel_occupancy(name##_kernel_of<E>(Lc, tk), wpb, smem, blocks);               \
  }
