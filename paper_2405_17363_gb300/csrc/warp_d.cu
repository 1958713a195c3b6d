// Instantiations of the warp-packed kernel for E = 13 14 15 16 rows per lane.
#include "warp_kernel.cuh"
#include "warp_launch.cuh"
namespace camp {
CAMP_KERNEL_DEFINE(warp, 13)
CAMP_KERNEL_DEFINE(warp, 14)
CAMP_KERNEL_DEFINE(warp, 15)
CAMP_KERNEL_DEFINE(warp, 16)
}  // namespace camp
