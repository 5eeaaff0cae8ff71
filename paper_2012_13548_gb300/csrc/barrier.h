// One look of a waiting block at a grid barrier (common.cuh, grid_sync), without the loads
// themselves, so that the order of the two reads can be tested on the host.
#pragma once

#ifdef __CUDACC__
#define GB_HD __host__ __device__ __forceinline__
#else
#define GB_HD inline
#endif

namespace gb {

enum BarrierLook { BARRIER_WAIT, BARRIER_PASSED, BARRIER_ERROR };

// arrived(): whether the counter has reached its target, an acquire; code(): the status word.
// A block that fails records its error before it arrives, or does not arrive, so the
// status counts only if it is read after the counter was seen full: then every error
// recorded before this barrier stops every block here, and no phase after it walks
// what a failed one left behind (a list's counter past the list's end).  While the
// counter is short the status read before it, in flight together with it, is enough to leave
// early; the second read is made once a barrier, when it has been passed.
template <typename Arrived, typename Code>
GB_HD BarrierLook barrier_look(Arrived arrived, Code code)
{
    const int early = code();
    const bool passed = arrived();
    if (early != 0) return BARRIER_ERROR;
    if (!passed) return BARRIER_WAIT;
    return code() != 0 ? BARRIER_ERROR : BARRIER_PASSED;
}

}  // namespace gb
