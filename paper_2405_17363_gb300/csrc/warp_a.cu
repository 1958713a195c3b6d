// Instantiations of the warp-packed kernel for E = 1 2 3 4 rows per lane.
#include "warp_kernel.cuh"
#include "warp_launch.cuh"
namespace camp {
CAMP_KERNEL_DEFINE(warp, 1)
CAMP_KERNEL_DEFINE(warp, 2)
CAMP_KERNEL_DEFINE(warp, 3)
CAMP_KERNEL_DEFINE(warp, 4)
}  // namespace camp
