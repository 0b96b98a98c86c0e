// K_chi, sum-tree form: launch plan and launcher (kernel in chi_lane.cuh).
#pragma once
#include "tissue_internal.h"

namespace tsg {

constexpr int kMaxSmem = 227 * 1024;  // dynamic shared memory a block may ask for
// Where a cell's voxels live during the step.
constexpr int kLeafShared = 0;   // shared memory: totals and 32-bit counts
constexpr int kLeafRecords = 1;  // scratch array: 64 bytes a quad, totals and packed counts
constexpr int kLeafSectors = 2;  // scratch array: 32 bytes a quad, its sum and 16-bit counts
constexpr int kLeafPlanes = 3;   // shared memory: three planes of 16-bit counts
// Shared leaves: R below this reads the Hill table unchecked (R + 1 too).
constexpr uint32_t kLaneHill = 2048;
constexpr uint32_t kWordCount = 1u << 19;    // counts of a record stay below
constexpr uint32_t kHalfCount = 0xFFFFu;     // ... of a sector or a plane, below what 16 bits hold

// First entry of level l of a four-ary tree whose levels follow one another:
// (4^l - 4) / 3.
__host__ __device__ constexpr uint32_t level_off(uint32_t l) {
  return (0x55555555u & ((1u << (2u * l)) - 1u)) - 1u;
}
// 64-bit words of sums a cell keeps in shared memory: cells of up to 4^lv
// voxels, G lanes each.  G < 8: a four-ary tree down to the quads (sectors: to
// four quads).  G >= 8: lane-wide nodes of R = 8 or 16 entries -- a root's copy,
// R nodes below it unless the root's entries are quads, and the quads' sums
// where those nodes' entries are four quads.
__host__ __device__ constexpr uint32_t lane_sum_words(int lv, int leaf, int G) {
  if (G < 8) return level_off(leaf == kLeafSectors ? lv - 1 : lv);
  const uint32_t R = G >= 16 ? 16u : 8u, under = (1u << (2 * lv)) / R;
  return R + (under > 4u ? R * R : 0u) + (under / R == 16u ? 256u : 0u);
}

// Shared memory that the two warps of a block with a helper exchange through.
constexpr uint32_t kExchangeBytes = 2 * 32 * (8 + 8 + 4 + 28) + 32 * 24 + 16;

struct LaneArgs {
  const TissueView* views;
  const uint2* items;  // (tissue, cell); nullptr: the cells of views[0] in order
  uint32_t* counter;   // work counter, zero before a launch of more cells than places
  uint64_t* scratch;   // the resident cells' records (plans with scratch_bytes > 0)
  uint2* redo;         // unless shared leaves: cells whose counts pass the packed range
  uint32_t* redo_n;
  double dt;
  uint32_t n_items, step_off;
  uint32_t V, n;       // of every listed cell
  uint32_t lut_bytes, cell_stride;
  uint64_t scratch_words;  // of `scratch` (read by the checked build)
};

struct LanePlan {
  uint32_t G = 0, wpb = 0, threads = 0, blocks = 0;  // G = 0: stays with the segmented kernel
  int leaf = kLeafShared;
  uint32_t helper = 0;    // blocks an SM of two warps, one of which draws ahead; 0: none
  uint32_t lut_bytes = 0, cell_stride = 0;
  size_t smem = 0, scratch_bytes = 0;
  bool small = false;     // at most one block per SM
  bool counters = false;  // the launch uses the work and redo counters (cleared before it)
};

// The plan for `cells` cells of V voxels; model 0: Notch-Delta without
// in-voxel binding, 1: Notch-Delta, 2: promoter.  `beside`: warps of launches
// that run at the same time and come first.
LanePlan lane_plan(uint32_t V, uint64_t cells, int model, uint64_t beside = 0);
cudaError_t launch_chi_lane(const LanePlan& plan, int model, const TissueView* d_views,
                            const uint2* d_items, uint32_t n_items, uint32_t* d_counter,
                            uint64_t* d_scratch, const ChiRedo& redo, uint32_t V, uint32_t n,
                            uint32_t step_off, double dt, cudaStream_t stream, int priority = 0,
                            bool early = false);
// What a launch of the plan, or of a shape of the segmented kernel, runs.
tissue_chi_info lane_info(const LanePlan& plan);
tissue_chi_info seg_info(const tissue_launch& shape, uint32_t V, int gen);
using ChiLaneKernel = void (*)(const LaneArgs);
// nullptr where not built.
// k_chi_lane.cu, k_chi_lane_bind.cu, k_chi_lane_pm.cu
ChiLaneKernel chi_lane_kernel_nd(uint32_t V, int leaf, uint32_t G, uint32_t helper);
ChiLaneKernel chi_lane_kernel_bind(uint32_t V, int leaf, uint32_t G, uint32_t helper);
ChiLaneKernel chi_lane_kernel_pm(uint32_t V, int leaf, uint32_t G, uint32_t helper);

}  // namespace tsg
