// Instantiations of the warp-packed kernel for E = 5 6 7 8 rows per lane.
#include "warp_kernel.cuh"
#include "warp_launch.cuh"
namespace camp {
CAMP_KERNEL_DEFINE(warp, 5)
CAMP_KERNEL_DEFINE(warp, 6)
CAMP_KERNEL_DEFINE(warp, 7)
CAMP_KERNEL_DEFINE(warp, 8)
}  // namespace camp
