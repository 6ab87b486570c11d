// step_slots.cuh -- which slot of the per-step counters a step counts in.
//
// Per-step counts live in four slots taken in turn: the steps of one kernel
// follow one another with as little as one grid barrier between them, so a
// block may already count the next step while another still reads this one's
// counts, and only the slot of the step before is free for everyone.  Each
// step clears that one after its first barrier.  Three slots would do; four
// divide the 2^32 values of a step number, which wraps round in a run of
// days, so that the turn goes on over the wrap, and a mask finds the slot of
// a negative number as well.
#pragma once

#ifdef __CUDACC__
#define LVB_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define LVB_HOST_DEVICE inline
#endif

namespace lvb {

constexpr int kStepSlots = 4;

// The number of the step after `done` steps, modulo 2^32.
LVB_HOST_DEVICE int next_step(unsigned done) { return (int)(done + 1u); }

LVB_HOST_DEVICE int step_slot(int step) { return step & (kStepSlots - 1); }
LVB_HOST_DEVICE int spent_slot(int slot) { return (slot + kStepSlots - 1) & (kStepSlots - 1); }

}  // namespace lvb
