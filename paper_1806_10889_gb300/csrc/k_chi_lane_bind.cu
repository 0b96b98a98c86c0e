// K_chi, sum-tree form: the instantiations for Notch-Delta with in-voxel binding (k_in, k_off).
// The kernel template is in chi_lane.cuh.
#include "chi_lane.cuh"

namespace tsg {

ChiLaneKernel chi_lane_kernel_bind(uint32_t V, int leaf, bool one) {
  if (V <= 64) {
    if (leaf == kLeafRecords) return one ? k_chi_lane<1, 3, kLeafRecords, true> : nullptr;
    return leaf == kLeafShared && !one ? k_chi_lane<1, 3, kLeafShared, false> : nullptr;
  }
  if (V <= 256) {
    if (leaf == kLeafRecords)
      return one ? k_chi_lane<1, 4, kLeafRecords, true> : k_chi_lane<1, 4, kLeafRecords, false>;
    return leaf == kLeafShared && !one ? k_chi_lane<1, 4, kLeafShared, false> : nullptr;
  }
  if (leaf == kLeafNodes)
    return one ? k_chi_lane<1, 5, kLeafNodes, true> : k_chi_lane<1, 5, kLeafNodes, false>;
  if (one) return nullptr;
  return leaf == kLeafRecords ? k_chi_lane<1, 5, kLeafRecords, false>
                              : k_chi_lane<1, 5, kLeafShared, false>;
}

}  // namespace tsg
