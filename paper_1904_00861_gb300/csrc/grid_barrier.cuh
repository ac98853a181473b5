// The barrier of the persistent (cooperative) loop kernels.
#pragma once

#include "bulk.cuh"
#include "dtsph_internal.cuh"

namespace dtsph {

// True when the arrival counter has reached target. Both wrap at 2^32 (steps of several
// million iterations) and lie less than 2^31 apart.
__host__ __device__ __forceinline__ bool barrier_reached(unsigned int arrivals, unsigned int target)
{
    return (int)(arrivals - target) >= 0;
}

// Grid barrier for a cooperative launch (all blocks resident): arrival counter
// `bar`, reset to 0 before the launch; the epoch-th barrier waits for
// epoch * gridDim.x arrivals: a release arrival of the block's writes, then polls.
// ALONE (one block per SM): acquire polls, the shortest way. Else relaxed polls and
// one acquire fence, since every acquire would empty the L1 under the SM's other
// blocks. The wait gives up after limit_ns (one second unless a test shortens it),
// raises kErrBarrier and returns false (the caller then stops iterating).
template <bool ALONE>
__device__ __forceinline__ bool grid_barrier(unsigned int *bar, unsigned int epoch, uint32_t *err, int &ok_sh,
                                             unsigned long long limit_ns)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int target = epoch * gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        int ok = 1, polls = 0;
        unsigned long long t0 = 0;
        for (;;) {
            unsigned int v;
            if (ALONE) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            else asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (barrier_reached(v, target)) break;
            // (the clock every 64 polls: reading it costs more than a poll)
            if (limit_ns == 0 || (++polls & 63) == 0) {
                const unsigned long long now = globaltimer_ns();
                if (t0 == 0) t0 = now;
                if (limit_ns == 0 || now - t0 > limit_ns) {
                    atomicOr(err, kErrBarrier);
                    ok = 0;
                    break;
                }
            }
        }
        if (!ALONE) asm volatile("fence.acq_rel.gpu;" ::: "memory");
        ok_sh = ok;
    }
    __syncthreads();
    return ok_sh != 0;
}

}  // namespace dtsph
