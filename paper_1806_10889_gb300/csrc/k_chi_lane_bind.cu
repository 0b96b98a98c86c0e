// K_chi, sum-tree form: the instantiations for Notch-Delta with in-voxel binding (k_in, k_off).
// The kernel template is in chi_lane.cuh.
#include "chi_lane.cuh"

namespace tsg {

ChiLaneKernel chi_lane_kernel_bind(uint32_t V, int leaf, bool one) {
  const int lv = V <= 64 ? 3 : V <= 256 ? 4 : 5;
  if (leaf == kLeafShared && !one)
    return lv == 3   ? k_chi_lane<1, 3, kLeafShared, false>
           : lv == 4 ? k_chi_lane<1, 4, kLeafShared, false>
                     : k_chi_lane<1, 5, kLeafShared, false>;
  if (leaf == kLeafRecords && lv == 3 && one) return k_chi_lane<1, 3, kLeafRecords, true>;
  if (leaf == kLeafRecords && lv == 4 && !one) return k_chi_lane<1, 4, kLeafRecords, false>;
  if (leaf == kLeafRecords && lv == 5 && !one) return k_chi_lane<1, 5, kLeafRecords, false>;
  if (leaf == kLeafSectors && lv == 4 && one) return k_chi_lane<1, 4, kLeafSectors, true>;
  if (leaf == kLeafSectors && lv == 5)
    return one ? k_chi_lane<1, 5, kLeafSectors, true> : k_chi_lane<1, 5, kLeafSectors, false>;
  return nullptr;
}

}  // namespace tsg
