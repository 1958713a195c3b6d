// Instantiations of the fused assembly + solve kernel
// for E = 1 2 3 4 rows per lane.
#include "warp_kernel.cuh"
#include "warp_launch.cuh"
namespace camp {
CAMP_KERNEL_DEFINE(assemble, 1)
CAMP_KERNEL_DEFINE(assemble, 2)
CAMP_KERNEL_DEFINE(assemble, 3)
CAMP_KERNEL_DEFINE(assemble, 4)
}  // namespace camp
