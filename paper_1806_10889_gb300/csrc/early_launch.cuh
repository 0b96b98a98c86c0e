// Early launches (programmatic dependent launch) of small tissues' steps.
//
// A step of a few cells is launches as much as events: 2x2 cells at dt 1e-9 take
// 20 us in three launches.  A kernel launched with the programmatic stream
// serialization attribute starts once every block of the launch before it has
// started, does what reads no device memory, and waits here for that launch to
// end: 15 us.  Only for tissues whose chi launch is at most one block per SM:
// blocks placed while the launch before still holds SMs spread unevenly (64x64
// cells, dt 0.01: 949 -> 1,095 us a step with all three launches early, 956 with
// the faces' alone).  6x4 cells of 16x16 voxels, dt 0.001: 91 -> 84 us a step.
#pragma once

namespace tsg {

// Let the next launch start, then wait for the one before (both at once when
// the launches are not early).
__device__ __forceinline__ void early_launch() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace tsg
