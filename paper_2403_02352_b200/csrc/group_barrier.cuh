// Barrier between the CTAs of a group inside a persistent cooperative kernel (all CTAs of the launch are resident).
#pragma once
#include "common.cuh"

constexpr unsigned SPIN_LIMIT = 1u << 22;

__device__ __forceinline__ void wait_ran_out(int *abort_flag)
{
    raise_status(abort_flag - 1, ATP_ERR_TIMEOUT);
    *(volatile int *)abort_flag = 1;
}

// Group barrier number `gen` (1, 2, ...) of a group of `ncta` CTAs: every CTA adds one to the arrival counter sync[0]
// (release) and polls the same word (acquire) until all have arrived. Polling the counter itself saves the hop through a
// second word that the last CTA to arrive would publish: 3400-3600 -> 2000 (18 CTAs) .. 2950 (296) cycles. A word per CTA, all
// polled by everybody, is no faster at 18 and 15700 cycles at 296; the counter spread over 4 or 8 lines is slower at every
// size. Bounded: returns false when the wait ran out or another CTA flagged an abort. abort_flag: the word after the device
// status; the CTA whose wait runs out records ATP_ERR_TIMEOUT there itself, because the others may find the barrier complete
// a moment later and finish without noticing. Data that crosses the barrier is read with L2 loads.
__device__ __forceinline__ bool group_barrier(unsigned *sync, unsigned gen, unsigned ncta, int *abort_flag,
                                              unsigned limit = SPIN_LIMIT)
{
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0 && ncta > 1) {
        // release / acquire at GPU scope: the block barrier above orders the CTA's writes before thread 0's
        // release, the one below orders its acquire before the CTA's later reads
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(sync) : "memory");
        ok = 0;
        for (unsigned i = 0; i < limit; ++i) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(sync) : "memory");
            if ((int)(v - gen * ncta) >= 0) { ok = 1; break; }
            if ((i & 1023u) == 1023u && *(volatile int *)abort_flag) break;
        }
        if (!ok) wait_ran_out(abort_flag);
    }
    return __syncthreads_and(ok) != 0;
}
