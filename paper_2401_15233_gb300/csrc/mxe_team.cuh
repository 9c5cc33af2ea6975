// mxe_team.cuh -- barrier of the CTAs that march one tube together, anywhere
// on the chip (a cooperative launch keeps all of them resident).
#pragma once
#include "mxe_internal.h"

namespace mxe {

// All threads of all `nb` CTAs; `target` counts arrivals since the launch.
// Returns false (in every thread of the CTA) if the wait gave up after `spin` polls.
__device__ __forceinline__ bool team_barrier(TubeSync* s, unsigned nb, unsigned& target, int spin) {
    __shared__ int ok;
    if (nb == 1u) {
        __syncthreads();
        return true;
    }
    target += nb;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();                       // the CTA's writes before its arrival
        atomicAdd(&s->count, 1u);
        int left = spin, good = 1;
        unsigned v;
        do {
            asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(&s->count) : "memory");
            if (--left == 0) {
                good = 0;
                break;
            }
        } while ((int)(v - target) < 0);
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

}  // namespace mxe
