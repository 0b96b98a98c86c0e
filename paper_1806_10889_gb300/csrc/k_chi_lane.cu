// K_chi, sum-tree form: the Notch-Delta instantiations, the launch plan and
// the launcher (the kernel template is in chi_lane.cuh).
#include "chi_lane.cuh"

namespace tsg {

ChiLaneKernel chi_lane_kernel_nd(uint32_t V, int leaf, uint32_t G, uint32_t helper) {
  return lane_instance<0>(V, leaf, G, helper);
}

namespace {

ChiLaneKernel lane_kernel(int model, uint32_t V, int leaf, uint32_t G, uint32_t helper) {
  return model == 2   ? chi_lane_kernel_pm(V, leaf, G, helper)
         : model == 1 ? chi_lane_kernel_bind(V, leaf, G, helper)
                      : chi_lane_kernel_nd(V, leaf, G, helper);
}

}  // namespace

// The shape follows from the cells an SM holds: the most lanes per cell with
// which one wave runs them all (12 or 16 warps an SM).  Few cells: one chain of
// events sets the time, and more lanes per cell take more of the draws off it.
// Many: the instructions issued per event do, and one lane per cell issues the
// fewest; past L2's size the random accesses to DRAM do, and a sector makes two
// reads and two writes an event.  Chi ms of one step at dt 0.02 (8x8 and 16x16
// voxels) and 0.006 (32x32), 60 D + 30 N + 10 R per voxel, by cells per SM; leaf
// (S shared, P planes, R records, X sectors) and lanes per cell; in parentheses
// the next shape, in brackets the segmented kernel's default launch:
//         8x8                          16x16                        32x32
//    4  S32 .26 (S16 .28) [.65]    S32 1.05 (S16 1.12) [2.6]    S32 1.39 (S16 1.43) [3.1]
//    6  S16 .29 (S32 .29) [.71]    S16 1.15 (S32 1.22) [2.8]    S16 1.48 (S32 1.60) [3.5]
//   12  S16 .34 (S8 .35)  [.79]    S16 1.34 (S8 1.36)  [3.1]    P16 1.92 (R16 2.68) [4.0]
//   24                           27 S8 1.68 (S4 2.10)  [4.1]    P16 2.47 (R16 3.3)  [6.1]
//   32  S8 .42  (S4 .54)  [.87]    S8 1.68  (S4 2.09)  [4.1]    R16 3.55 (R8 4.03)  [6.7]
//   48  S8 .52  (S4 .63)  [.98]  44 P8 2.28 (R8 2.93)  [5.2]  33 R8 4.26 (R16 5.5)  [9.8]
//   64  S4 .63  (S8 .91)  [1.2]    P8 2.82  (R8 3.36)  [6.1]    R8 5.13  (X1 6.4)  [13.3]
//   88  S4 .76  (R1 1.15) [2.0]    P4 3.25  (R4 4.1)   [9.7]  65 X1 6.45 (R8 7.7)  [15.2]
//  128  P4 .92  (R1 1.06) [2.2]    R4 4.58  (X1 5.24) [12.1]
//  150  R1 1.12 (R4 1.36) [2.8]    X1 5.17  (R4 7.2)  [15.0]    X1 8.2             [30.1]
//  431  R1 1.79           [7.0]    X1 9.0             [39.1]    X1 18.1            [84.0]
// Cells of 10x10 voxels fit shared memory longer: 50 to 64 an SM take S4 (.98,
// R8 1.13 to 1.20), 81 to 128 P4.
LanePlan lane_plan(uint32_t V, uint64_t cells, int model, uint64_t beside) {
  LanePlan pl;
  int dev = 0, sms = 0;
  if (cells == 0 || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return pl;
  const int lv = V <= 64 ? 3 : V <= 256 ? 4 : 5;
  const uint64_t per = (cells + static_cast<uint64_t>(sms) - 1) / static_cast<uint64_t>(sms);
  const uint32_t G = per <= 4                       ? 32u
                     : per <= (lv == 5 ? 32u : 12u) ? 16u
                     : per <= (lv == 3 ? 48u : 64u) ? 8u
                     : per <= 128 && lv < 5         ? 4u
                                                    : 1u;
  // A helper warp that draws ahead while at most eight warps an SM run cells: the
  // draws leave the chain.  Up to six, twelve warps have the registers they want
  // (168).  Chi ms, without -> with: 2x2 cells of 8x8 voxels 1.19 -> 1.14, 60x50 of
  // 16x16 8.34 -> 7.70, 60 uneven tissues (26,802 cells of 32x32) 146.7 -> 133.9.
  // One lane per cell, 190 cells of 16x16 an SM: 5.81 -> 5.24.
  // Seven and eight leave 128: 64x64 of 16x16 9.35 -> 9.12, promoter 7.41 -> 6.95,
  // 64x64 of 8x8 3.83 -> 3.69, 48x48 of 32x32 (records, then) 45.05 -> 44.36; with
  // in-voxel binding the spills cost more (16x16 9.74 -> 10.01) and it is not
  // built for 8 lanes; below six warps 128 registers cost 2% (7.68 -> 7.81).
  // Classes of a batch share the SMs, the first ahead of the others, which run
  // in what it leaves: a helper there takes warps and issue slots from it (60
  // uneven tissues, helpers in all three classes 138.8, with this count 132.9).
  const uint64_t runs = beside + (cells * G + 31u) / 32u;
  const uint32_t few = runs <= 6u * static_cast<uint64_t>(sms)   ? 6u
                       : runs <= 8u * static_cast<uint64_t>(sms) ? 8u
                                                                 : 0u;
  const uint32_t nq = (V + 3u) / 4u;
  int per_sm = 0;  // blocks an SM holds
  // Leaves: in shared memory while one wave of cells fits there (the shortest
  // chain, also with four lanes per cell instead of eight); else as planes there
  // (cells of 16x16, 37 to 64 an SM: planes 2.28 to 2.82 ms, records 2.9 to 3.4;
  // where S8 fits, 2.09); else records, whose totals need no recomputing, in the scratch
  // array; for one lane per cell, where L2's size and the
  // sums in shared memory (2.7 KB a cell of 32x32 voxels) bound the cells in
  // flight, sectors: half the bytes and a quarter of the sums (8x8 keeps records,
  // 9.0 against 10.7 ms for 256x256 cells).
  auto shape = [&](uint32_t G, int leaf, uint32_t helper) {
    const uint64_t places = 32u / G;  // cells a warp runs
    pl.G = G;
    const uint32_t cell = 48u + 8u * lane_sum_words(lv, leaf, static_cast<int>(G)) +
                          (leaf == kLeafShared ? 80u : leaf == kLeafPlanes ? 24u : 0u) * nq;
    // an odd multiple of 16 bytes: lanes reading the same entry of their cells
    // start on different shared-memory banks
    pl.cell_stride = ((cell + 15u) & ~15u) | 16u;
    pl.lut_bytes = 128u + 16u * ((nq + 3u) / 4u) + (helper ? kExchangeBytes : 0u);
    pl.leaf = leaf;
    pl.helper = helper;
    pl.wpb = G == 1 && !helper ? 2u : 1u;
    pl.threads = helper ? 64u : 32u * pl.wpb;
    pl.smem = pl.lut_bytes + static_cast<size_t>(pl.wpb * places) * pl.cell_stride;
    // The answer: whether one wave holds every cell.  The shared-memory limit is
    // the device's, not this plan's: plans of other cell sizes share the kernel.
    const ChiLaneKernel k = lane_kernel(model, V, leaf, G, helper);
    per_sm = 0;
    if (!k || pl.smem > kMaxSmem ||
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, static_cast<int>(pl.threads),
                                                      pl.smem) != cudaSuccess)
      per_sm = 0;
    return per <= static_cast<uint64_t>(per_sm) * pl.wpb * places;
  };
  // A helper is asked for first.
  auto fits = [&](uint32_t G, int leaf) {
    return (few && shape(G, leaf, few)) || shape(G, leaf, 0);
  };
  // The first form, in the order above, that holds all cells; one that holds some
  // of them if none does.
  auto any_form = [&](uint32_t G) {
    return fits(G, kLeafShared) || (G == 8 && shape(4, kLeafShared, 0)) || fits(G, kLeafPlanes) ||
           fits(G, G == 1 && lv > 3 ? kLeafSectors : kLeafRecords) || per_sm >= 1 ||
           (shape(G, kLeafShared, 0), per_sm >= 1);
  };
  // A small class beside others that leave no helper: up to 256 voxels 32 and 16
  // lanes without one, whose blocks are the smallest and find room beside the
  // first class's (1,500 cells of 32x32 with 500 of 16x16 and 500 of 8x8: the chi
  // phase 11.1 ms, with 8 lanes 13.8, with the segmented kernel 10.8; 3,500 of
  // 16x16 with 500 of 15x15: 4.1, 5.8, 6.4).  Above, 32 lanes take 25 KB a cell and
  // wait for the first class to end (6,400 of 32x32 with 400 of 31x31: 30.0 ms):
  // not built, the next narrower form, planes, takes them (25.0; segmented 25.8; beside
  // 1,600 of 32x32 20.9, 23.2 and 34.9).
  for (uint32_t g = G; g >= 1u && !any_form(g);) g /= 2u;
  if (per_sm < 1) {
    pl.G = 0;
    return pl;
  }
  const uint64_t per_block = static_cast<uint64_t>(pl.wpb) * (32u / pl.G);
  const uint64_t need = (cells + per_block - 1) / per_block;
  const uint64_t cap = static_cast<uint64_t>(sms) * static_cast<uint64_t>(per_sm);
  pl.blocks = static_cast<uint32_t>(need < cap ? need : cap);
  pl.small = need <= static_cast<uint64_t>(sms);
  pl.counters = need > cap || pl.leaf != kLeafShared;
  if (pl.leaf == kLeafRecords || pl.leaf == kLeafSectors)
    pl.scratch_bytes = static_cast<size_t>(pl.blocks) * per_block *
                       (pl.leaf == kLeafRecords ? 8u * nq : 16u * ((nq + 3u) / 4u)) *
                       sizeof(uint64_t);
  return pl;
}

tissue_chi_info lane_info(const LanePlan& pl) {
  return tissue_chi_info{1, pl.G, pl.leaf == kLeafShared ? 1u : 2u, 0, pl.scratch_bytes};
}

tissue_chi_info seg_info(const tissue_launch& c, uint32_t V, int gen) {
  const int H = static_cast<int>(c.lanes_per_cell);
  const bool narrow = c.kernel == TISSUE_KERNEL_PERSISTENT && gen == 0 && V > 256 &&
                      chi_seg_kernel_narrow(H, c.smem_layout == TISSUE_LAYOUT_PREFIX,
                                            V > static_cast<uint32_t>(H * H));
  return tissue_chi_info{0, c.lanes_per_cell, narrow ? 2u : 1u, 0, 0};
}

cudaError_t launch_chi_lane(const LanePlan& pl, int model, const TissueView* d_views,
                            const uint2* d_items, uint32_t n_items, uint32_t* d_counter,
                            uint64_t* d_scratch, const ChiRedo& redo, uint32_t V, uint32_t n,
                            uint32_t step_off, double dt, cudaStream_t stream, int priority,
                            bool early) {
  const ChiLaneKernel k = lane_kernel(model, V, pl.leaf, pl.G, pl.helper);
  const LaneArgs a{d_views, d_items, d_counter, d_scratch, redo.items, redo.counters + 1, dt,
                   n_items, step_off, V, n, pl.lut_bytes, pl.cell_stride,
                   pl.scratch_bytes / sizeof(uint64_t)};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl.blocks);
  cfg.blockDim = dim3(pl.threads);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributePriority;
  attr[0].val.priority = priority;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  // the priority, if there is one, and the early start
  cfg.attrs = priority ? attr : attr + 1;
  cfg.numAttrs = (priority ? 1u : 0u) + (early ? 1u : 0u);
  cudaError_t e = cudaLaunchKernelEx(&cfg, k, a);
  if (e != cudaSuccess || pl.leaf == kLeafShared) return e;
  // the cells that left the packed range, by the segmented kernel from the
  // state they started the step with (it reads their number from the device, and
  // does not wait for the launch before: never early)
  cfg.attrs = attr;
  cfg.numAttrs = priority ? 1 : 0;
  // in the shape that kernel has by default for as many cells: where every cell is
  // past the packed range, the time it takes alone (N at 70,000 a voxel, 256x180
  // cells of 16x16 voxels 59.9 -> 50.0 ms against the prefix layout, 128x160 of
  // 32x32 88.5 -> 70.8)
  tissue_launch c = default_launch(V, n_items);
  if (c.smem_layout == TISSUE_LAYOUT_RECOMPUTE &&
      !recompute_covers(V, static_cast<int>(c.lanes_per_cell), model == 2 ? 2 : 0))
    c = prefix_launch(V, n_items);
  const int H = static_cast<int>(c.lanes_per_cell);
  const bool qb = V > static_cast<uint32_t>(H * H), pre = c.smem_layout == TISSUE_LAYOUT_PREFIX;
  const ChiSegKernel ks =
      model == 2 ? chi_seg_kernel_pm(H, pre, qb) : chi_seg_kernel_nd(H, pre, qb);
  const uint32_t seg_bytes = seg_bytes_for(V, H, pre);
  const size_t smem = static_cast<size_t>(c.warps_per_block) * (32u / c.lanes_per_cell) * seg_bytes;
  const int threads = 32 * static_cast<int>(c.warps_per_block);
  int dev = 0, sms = 0, per_sm = 0;
  if (smem > 48 * 1024 &&
      (e = cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(smem))) != cudaSuccess)
    return e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ks, threads, smem)) != cudaSuccess)
    return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  cfg.gridDim = dim3(static_cast<unsigned>(sms * per_sm));
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  return cudaLaunchKernelEx(&cfg, ks, d_views, static_cast<const uint2*>(redo.items), n_items,
                            redo.counters + 2, seg_bytes, step_off, dt,
                            static_cast<uint2*>(nullptr), static_cast<uint32_t*>(nullptr),
                            static_cast<const uint32_t*>(redo.counters + 1));
}

}  // namespace tsg
