// Instantiations of the fused assembly + solve kernel
// for E = 5 6 7 8 rows per lane.
#include "warp_kernel.cuh"
#include "warp_launch.cuh"
namespace camp {
CAMP_KERNEL_DEFINE(assemble, 5)
CAMP_KERNEL_DEFINE(assemble, 6)
CAMP_KERNEL_DEFINE(assemble, 7)
CAMP_KERNEL_DEFINE(assemble, 8)
}  // namespace camp
