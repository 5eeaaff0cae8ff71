// Shared device helpers of the GB300 Graph500 library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "barrier.h"
#include "gb300bfs.h"
#include "internal.h"

namespace gb {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------
// Device status word: the first error a kernel records wins; nothing traps.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void record_error(DevStatus *st, int code, int where, long long detail)
{
    if (atomicCAS(&st->code, 0, code) == 0) {
        st->where = where;
        st->detail = detail;
    }
}

__device__ __forceinline__ int status_code(const DevStatus *st)
{
    return *(volatile const int *)&st->code;
}

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t ld_acquire_u64(const unsigned long long *p)
{
    uint64_t v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned ld_volatile_u32(const unsigned *p)
{
    return *(volatile const unsigned *)p;
}

// Sites of kernel 1's input errors (DevStatus::where): an endpoint, a weight.
constexpr int SITE_K1_RANGE = 10, SITE_SP_W = 45;

// Weight w in (0, 1] as units of 2^-24, rounded to the nearest unit and at
// least one; 0 for a weight outside (0, 1] or NaN.
__device__ __forceinline__ uint32_t weight_units(float w)
{
    if (!(w > 0.0f && w <= 1.0f)) return 0u;
    const uint32_t k = __float2uint_rn(w * 16777216.0f);
    return k < 1u ? 1u : k;
}

// ---------------------------------------------------------------------------
// Software grid barrier for cooperative (all-blocks-resident) launches.
// Arrivals only ever add to one counter: the k-th barrier of a launch is
// passed once the counter reaches base + k * gridDim.x, so no block has to
// reset anything and the last arrival frees the others directly.  Thread 0
// arrives with a release add (after __syncthreads, it publishes the block's
// writes) and waits with acquire loads.  Every wait is bounded by
// `timeout_ns` of the global timer: on expiry the block records
// GB_ERR_TIMEOUT, and every block leaves early once any block has recorded an
// error; grid_sync then returns false.  An error recorded before a barrier (with
// grid_error) stops every block at that barrier at the latest (barrier.h).
// ---------------------------------------------------------------------------
struct GridBarrier {
    unsigned long long word;
    unsigned pad[30];  // a line of its own: the blocks that wait read it all the time, beside
                       // the atomics on the level's counters of the blocks still at work
};

__device__ __forceinline__ void red_release_add_u64(unsigned long long *p, uint64_t v)
{
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// What thread 0 of a block keeps of the barrier, in shared memory: as registers of every
// thread for the whole kernel it made the searches spill.
struct BlockBarrier {
    BarrierState state;
    int failed;  // a thread of this block has recorded an error in this launch
};
__device__ __forceinline__ BlockBarrier &block_barrier()
{
    __shared__ BlockBarrier s_bar;
    return s_bar;
}

// record_error in a kernel with grid barriers.
__device__ __forceinline__ void grid_error(DevStatus *st, int code, int where, long long detail)
{
    block_barrier().failed = 1;
    record_error(st, code, where, detail);
}

// Call once at kernel entry, before the block's first grid_sync and grid_error.  No
// kernel records an error before its first barrier but by not arriving there, so the
// error count is the earlier launches'.
__device__ __forceinline__ void grid_barrier_begin(GridBarrier *b)
{
    if (threadIdx.x == 0) {
        block_barrier().state = barrier_start(ld_acquire_u64(&b->word), gridDim.x);
        block_barrier().failed = 0;
    }
    __syncthreads();
}

__device__ __forceinline__ bool grid_sync(GridBarrier *b, DevStatus *st, uint64_t timeout_ns, int site)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        red_release_add_u64(&b->word, barrier_arrival(block_barrier().failed != 0));
        BarrierState state = block_barrier().state;
        state.target += gridDim.x;
        block_barrier().state.target = state.target;
        uint64_t t0 = 0;
        unsigned spins = 0;
        for (;;) {
            const BarrierLook look =
                barrier_look(state, [&] { return status_code(st); }, [&] { return ld_acquire_u64(&b->word); });
            if (look == BARRIER_ERROR) ok = 0;
            if (look != BARRIER_WAIT) break;
            // the clock from the first poll on, every eighth: a poll is an L2 round
            // trip, so a limit below a few microseconds runs out within them
            if ((++spins & 7u) == 1) {
                const uint64_t now = globaltimer_ns();
                if (t0 == 0) {
                    t0 = now;
                } else if (now - t0 > timeout_ns) {
                    record_error(st, GB_ERR_TIMEOUT, site, (long long)blockIdx.x);
                    ok = 0;
                    break;
                }
            }
            __nanosleep(32);
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// ---------------------------------------------------------------------------
// Warp helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// inclusive prefix sum across the warp
template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v)
{
    const unsigned lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(kFull, v, o);
        if (lane >= (unsigned)o) v += t;
    }
    return v;
}

// How many of `cnt` rows a warp takes at a time: 32 if that leaves none of
// `nwarps` warps without, else fewer.  A warp streams its rows' edges in rounds of
// dependent memory accesses, 2-3 us each, and a level lasts as long as its longest
// warp: 32 rows of up to 256 entries in one warp while thousands had none were half of
// a wide level's time.
__device__ __forceinline__ int rows_per_warp(int64_t cnt, int64_t nwarps)
{
    return cnt >= 32 * nwarps ? 32 : (int)((cnt + nwarps - 1) / nwarps);
}

// Loads that bypass L1: data written by other blocks of the same kernel.
__device__ __forceinline__ unsigned ldcg_u32(const unsigned *p) { return __ldcg(p); }
__device__ __forceinline__ int ldcg_i32(const int *p) { return __ldcg(p); }
__device__ __forceinline__ unsigned long long ldcg_u64(const unsigned long long *p)
{
    return __ldcg(p);
}

// A hint (TMA bulk prefetch) that brings `bytes` bytes at p into L2; it
// neither waits nor changes any value.  p and bytes must be multiples of 16
// and the range must lie inside one allocation.
__device__ __forceinline__ void prefetch_l2_bulk(const void *p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

}  // namespace gb
