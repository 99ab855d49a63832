// lbm_barrier.cuh -- the bounded grid barrier of the cooperative launches.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {

// Arrive and wait until `expected` CTAs have arrived (bounded).  Returns
// false (and sets ERR_TIMEOUT in *err) if the wait gave up.
__device__ __forceinline__ bool grid_barrier(GridBarrier *bar, unsigned expected, long long budget, uint32_t *err)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        volatile unsigned *vg = &bar->gen;
        volatile uint32_t *ve = err;
        const unsigned g = *vg;
        __threadfence();   // this CTA's stores (ordered by the CTA barrier) before the arrival
        if (atomicAdd(&bar->count, 1u) == expected - 1) {
            atomicExch(&bar->count, 0u);
            __threadfence();
            atomicAdd(&bar->gen, 1u);
        } else {
            const long long t0 = clock64();
            while (*vg == g) {
                if ((*ve & ERR_TIMEOUT) || clock64() - t0 > budget) {
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
        __threadfence();   // the other CTAs' stores before this CTA's next loads
        if (!ok) atomicOr(err, (uint32_t)ERR_TIMEOUT);
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

}  // namespace lbm
