// Which warp issues which use of the INT4 GEMM's TMEM slots (gemm_w4a4_kernel.cuh).  Plain C++, no CUDA types.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define W4A4_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define W4A4_HOST_DEVICE inline
#endif

namespace w4a4 {

constexpr int kTmemSlots = 2;   // one per group in flight

// A code-MMA warp's place in the sequence of slot uses, in which use u takes slot u % 2: per tile the low-rank entry, if there is one,
// and then the groups.  Two warps share the sequence by slot: each issues every use of its own slot and none of the other's, so it
// waits for every release of that slot, in order.  An mbarrier's parity tells a phase from the next one only: a warp that merely
// watches a use it does not issue can poll when the others are already two phases further, and then waits for good.  (Shared by
// the groups of a stage instead, with both warps waiting for a tile's first use, that was the case after a poll that came late.)
struct CodeSlotWalk {
  uint32_t own;         // this warp's slot
  uint32_t next = 0;    // the slot of the next use in the sequence
  uint32_t phase = 0;   // its slot is free once the phase of parity `phase ^ 1` has completed
  W4A4_HOST_DEVICE explicit CodeSlotWalk(uint32_t slot) : own(slot) {}
  W4A4_HOST_DEVICE bool owns_next() const { return next == own; }
  W4A4_HOST_DEVICE uint32_t group() const { return next ^ own; }   // which of a stage's two groups falls on the slot, as seen at the stage's start
  W4A4_HOST_DEVICE uint32_t free_parity() const { return phase ^ 1u; }
  W4A4_HOST_DEVICE void issued() { phase ^= 1u; }                  // a use of its slot
  W4A4_HOST_DEVICE void pass(uint32_t uses) { next ^= uses & 1u; }   // that many uses of the sequence, its own among them
};

}  // namespace w4a4
