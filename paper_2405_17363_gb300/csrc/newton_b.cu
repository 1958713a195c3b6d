// Instantiations of the device Newton corrector (rates, fused assembly and solve per iteration)
// for E = 5 6 7 8 rows per lane.
#include "warp_kernel.cuh"
#include "warp_launch.cuh"
namespace camp {
CAMP_KERNEL_DEFINE(newton, 5)
CAMP_KERNEL_DEFINE(newton, 6)
CAMP_KERNEL_DEFINE(newton, 7)
CAMP_KERNEL_DEFINE(newton, 8)
}  // namespace camp
