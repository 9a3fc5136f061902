// Progress of a column pass over its rows, in a word of global memory: a pass of one warp writes
// its boundary column row group by row group and publishes how many are written; the warp of
// the next pass waits until the groups it is about to read are there.  A wait only ever points
// at a pass whose warp is running: the passes of a task are handed out in order by one ticket.  So
// it ends, whichever other CTAs are resident; it is bounded all the same.
#pragma once
#include <cstdint>

#include "cm_internal.h"

namespace cm {
namespace {

// waits (lane 0 polls) until `need` row groups are written; false on every lane once `limit`
// polls have passed, or when another wait has given up and set `err`.  Lane 0's acquire orders
// only what lane 0 does next; the barrier after it passes that order on to the lanes that read
// the rows (a shuffle does not).
__device__ __forceinline__ bool wait_groups(const int32_t* done, int32_t need, const int32_t* err,
                                            int32_t limit = kPollLimit)
{
    int ok = 1;
    if ((threadIdx.x & 31) == 0) {
        for (int polls = 0;; ++polls) {
            int32_t v;
            asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
            if (v >= need) break;
            if (polls >= limit ||
                ((polls & 1023) == 1023 && *reinterpret_cast<const volatile int32_t*>(err) != 0)) {
                ok = 0;
                break;
            }
            __nanosleep(100);
        }
    }
    __syncwarp();
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

__device__ __forceinline__ void publish_groups(int32_t* done, int32_t groups)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(done), "r"(groups) : "memory");
}

}  // namespace
}  // namespace cm
