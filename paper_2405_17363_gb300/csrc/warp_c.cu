// Instantiations of the warp-packed kernel for E = 9 10 11 12 rows per lane.
#include "warp_kernel.cuh"
#include "warp_launch.cuh"
namespace camp {
CAMP_KERNEL_DEFINE(warp, 9)
CAMP_KERNEL_DEFINE(warp, 10)
CAMP_KERNEL_DEFINE(warp, 11)
CAMP_KERNEL_DEFINE(warp, 12)
}  // namespace camp
