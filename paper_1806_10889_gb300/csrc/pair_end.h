// The end of a block of two warps that meet at one barrier a batch: the warp
// that runs cells announces the batch at which it stops, the helper asks for it
// after that batch's barrier and before anything else.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define TSG_BOTH __host__ __device__ __forceinline__
#else
#define TSG_BOTH inline
#endif

namespace tsg {

// One flag for even and one for odd batches.  The running warp writes the flag
// of the batch whose barrier comes next; a helper that has passed the barrier
// before it but has not asked yet asks for the other one.  With a single flag
// such a helper would see the end one batch early and leave, and the running
// warp would wait at the last barrier for a warp that is gone.  A flag is
// written again two barriers later at the earliest, which the helper reaches
// only after it has asked.
struct PairEnd {
  int at[2];
  TSG_BOTH void clear() { at[0] = at[1] = 0; }
  TSG_BOTH void announce(uint32_t phase) { at[phase & 1u] = 1; }     // before the phase's barrier
  TSG_BOTH bool reached(uint32_t phase) const { return at[phase & 1u] != 0; }  // after it
};

}  // namespace tsg
