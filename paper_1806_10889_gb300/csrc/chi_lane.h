// K_chi, sum-tree form: launch plan and launcher (kernel in chi_lane.cuh).
#pragma once
#include "tissue_internal.h"

namespace tsg {

constexpr int kMaxSmem = 227 * 1024;  // dynamic shared memory a block may ask for
// Where a cell's voxels live during the step.
constexpr int kLeafShared = 0;   // shared memory: totals and 32-bit counts
constexpr int kLeafRecords = 1;  // scratch array: 64 bytes a quad, totals and packed counts
constexpr int kLeafSectors = 2;  // scratch array: 32 bytes a quad, its sum and 16-bit counts
constexpr uint32_t kLaneHill = 2048;  // R below this reads the Hill table unchecked (R + 1 too)
constexpr uint32_t kWordCount = 1u << 19;    // counts of a record stay below
constexpr uint32_t kSectorCount = 1u << 16;  // counts of a sector

struct LaneArgs {
  const TissueView* views;
  const uint2* items;  // (tissue, cell); nullptr: the cells of views[0] in order
  uint32_t* counter;   // work counter, zero before the launch
  uint64_t* scratch;   // the resident cells' records (plans with scratch_bytes > 0)
  uint2* redo;         // with records: cells whose counts pass the packed range
  uint32_t* redo_n;
  double dt;
  uint32_t n_items, step_off;
  uint32_t V, n;       // of every listed cell
  uint32_t G;          // lanes per cell
  uint32_t lut_bytes, cell_stride;
};

struct LanePlan {
  uint32_t G = 0, wpb = 0, blocks = 0;  // G = 0: this launch stays with the segmented kernel
  int leaf = kLeafShared;
  uint32_t lut_bytes = 0, cell_stride = 0;
  size_t smem = 0, scratch_bytes = 0;
};

// The plan for `cells` cells of V voxels; model 0: Notch-Delta without
// in-voxel binding, 1: Notch-Delta, 2: promoter.
LanePlan lane_plan(uint32_t V, uint64_t cells, int model);
cudaError_t launch_chi_lane(const LanePlan& plan, int model, const TissueView* d_views,
                            const uint2* d_items, uint32_t n_items, uint32_t* d_counter,
                            uint64_t* d_scratch, const ChiRedo& redo, uint32_t V, uint32_t n,
                            uint32_t step_off, double dt, cudaStream_t stream, int priority = 0);
using ChiLaneKernel = void (*)(const LaneArgs);
// one: G = 1; nullptr where not built.
ChiLaneKernel chi_lane_kernel_nd(uint32_t V, int leaf, bool one);      // k_chi_lane.cu
ChiLaneKernel chi_lane_kernel_bind(uint32_t V, int leaf, bool one);    // k_chi_lane_bind.cu
ChiLaneKernel chi_lane_kernel_pm(uint32_t V, int leaf, bool one);      // k_chi_lane_pm.cu

}  // namespace tsg
