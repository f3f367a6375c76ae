// Barrier over all CTAs of a cooperative launch (co-resident by its guarantee), with a bounded wait.
#pragma once
#include <cuda_runtime.h>

#include <cstdlib>

#include "../../include/dfhf.h"

namespace dfhf {

constexpr long long GRID_WAIT_CYCLES = 4000000000LL;   // about 2 s

// Budget of a barrier's wait: GRID_WAIT_CYCLES, or DFHF_GRID_WAIT_CYCLES (a test knob that makes the waits run out,
// to exercise the DF_E_TIMEOUT path)
inline long long grid_wait_cycles() {
    const char* v = std::getenv("DFHF_GRID_WAIT_CYCLES");
    const long long c = v ? std::atoll(v) : 0;
    return (c > 0 && c < GRID_WAIT_CYCLES) ? c : GRID_WAIT_CYCLES;
}

// count: arrivals, zero at the start of the launch; target: this CTA's running target, zero at the start; wait: the
// budget in cycles. False on every thread if the wait expires here or err is set elsewhere. What a CTA wrote before
// the barrier is visible to every CTA after it.
__device__ inline bool grid_barrier(unsigned* count, int* err, unsigned& target, long long wait) {
    __shared__ int ok;
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
        int good = 1;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(count) : "memory");
        const long long t0 = clock64();
        // arrivals only grow; the difference is taken modulo 2^32
        for (;;) {
            unsigned seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(seen) : "l"(count) : "memory");
            if ((int)(seen - target) >= 0) break;
            if (clock64() - t0 > wait || *(volatile int*)err) {
                atomicExch(err, DF_E_TIMEOUT);
                good = 0;
                break;
            }
        }
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

}  // namespace dfhf
