// K_chi, sum-tree form: the instantiations for Notch-Delta with in-voxel binding (k_in, k_off).
// The kernel template is in chi_lane.cuh.
#include "chi_lane.cuh"

namespace tsg {

ChiLaneKernel chi_lane_kernel_bind(uint32_t V, int leaf, uint32_t G, uint32_t helper) {
  return lane_instance<1>(V, leaf, G, helper);
}

}  // namespace tsg
