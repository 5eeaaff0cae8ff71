// One look of a waiting block at a grid barrier (common.cuh, grid_sync), without the loads
// themselves, so that what it concludes from them can be tested on the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GB_HD __host__ __device__ __forceinline__
#else
#define GB_HD inline
#endif

namespace gb {

enum BarrierLook { BARRIER_WAIT, BARRIER_PASSED, BARRIER_ERROR };

// The barrier's word: arrivals in its lower 48 bits (a word that serves many launches
// counts on: 32 bits were full after some minutes of serving, and 2^32 is no multiple of
// the grid), above them how many came from blocks that had recorded an error.
constexpr int kBarrierErrors = 48;
GB_HD uint64_t barrier_arrival(bool failed) { return 1u | ((uint64_t)failed << kBarrierErrors); }

// What a block has to reach: the arrivals of its next barrier (their low bits are enough
// to compare), and the error count that its launch began with.
struct BarrierState {
    unsigned target, errors;
};
// Before the first barrier of a launch of `blocks` blocks on a word: the multiple of the
// grid that earlier launches, which passed all their barriers, have left.
GB_HD BarrierState barrier_start(uint64_t word, unsigned blocks)
{
    const uint64_t arrivals = word & ((uint64_t(1) << kBarrierErrors) - 1);
    return {(unsigned)(arrivals / blocks * blocks), (unsigned)(word >> kBarrierErrors)};
}

// code(): the status word; word(): the barrier's word, an acquire.  Every error recorded
// before the barrier arrives with its block, in the word that says the barrier is
// complete, so it stops every block here and no phase after it walks what a failed one left
// behind (a list's counter past the list's end).  The status word, read in flight together
// with the other, only lets a block leave early: a block that timed out never
// arrives.  Reading the status once more after the word instead cost one more
// L2 latency a barrier: eight SCALE 20 searches 773 -> 790 us (so 776), SCALE 22 shortest
// paths 3.75 -> 3.80 ms (so 3.74), SCALE 10 searches 1.5 us of 46 (so 0.5).
template <typename Code, typename Word>
GB_HD BarrierLook barrier_look(const BarrierState &b, Code code, Word word)
{
    const int early = code();
    const uint64_t w = word();
    if (early != 0) return BARRIER_ERROR;
    if ((int)((unsigned)w - b.target) < 0) return BARRIER_WAIT;
    return (unsigned)(w >> kBarrierErrors) != b.errors ? BARRIER_ERROR : BARRIER_PASSED;
}

}  // namespace gb
