// K_chi, sum-tree form: the instantiations for the promoter model.
// The kernel template is in chi_lane.cuh.
#include "chi_lane.cuh"

namespace tsg {

ChiLaneKernel chi_lane_kernel_pm(uint32_t V, int leaf, bool one) {
  if (V <= 64) {
    if (leaf == kLeafRecords) return one ? k_chi_lane<2, 3, kLeafRecords, true> : nullptr;
    return leaf == kLeafShared && !one ? k_chi_lane<2, 3, kLeafShared, false> : nullptr;
  }
  if (V <= 256) {
    if (leaf == kLeafRecords)
      return one ? k_chi_lane<2, 4, kLeafRecords, true> : k_chi_lane<2, 4, kLeafRecords, false>;
    return leaf == kLeafShared && !one ? k_chi_lane<2, 4, kLeafShared, false> : nullptr;
  }
  if (leaf == kLeafNodes)
    return one ? k_chi_lane<2, 5, kLeafNodes, true> : k_chi_lane<2, 5, kLeafNodes, false>;
  if (one) return nullptr;
  return leaf == kLeafRecords ? k_chi_lane<2, 5, kLeafRecords, false>
                              : k_chi_lane<2, 5, kLeafShared, false>;
}

}  // namespace tsg
