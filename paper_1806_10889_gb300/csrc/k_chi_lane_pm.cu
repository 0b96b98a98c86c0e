// K_chi, sum-tree form: the instantiations for the promoter model.
// The kernel template is in chi_lane.cuh.
#include "chi_lane.cuh"

namespace tsg {

ChiLaneKernel chi_lane_kernel_pm(uint32_t V, int leaf, uint32_t G, uint32_t helper) {
  return lane_instance<2>(V, leaf, G, helper);
}

}  // namespace tsg
