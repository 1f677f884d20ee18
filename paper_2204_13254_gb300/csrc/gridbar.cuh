// Grid barrier of the cooperative vector kernels (gmres.cu, kernels.cu).
#pragma once

#include <cstdint>

namespace {

constexpr unsigned kMeetPolls = 1u << 19;   // of one barrier wait (about half a second)

// Grid barrier at a counter that is zero at its first arrival; false, in every thread, when it
// gave up (then *err is set).  *failed, in shared memory, is thread 0's: before the kernel's
// first barrier PcgScalars::wait_first (> 0 makes that barrier wait, this many polls long, for
// an arrival that nobody makes), afterwards 0 or 1.
__device__ bool grid_meet(uint32_t* ctr, int32_t* err, int* failed) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(ctr, 1u);
        const int first = *failed;
        const uint32_t all = gridDim.x + (first > 0 ? 1u : 0u);
        const unsigned limit = first > 0 ? (unsigned)first : kMeetPolls;
        unsigned k = 0;
        uint32_t v;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        } while (v < all && ++k < limit);
        *failed = v < all;
        if (*failed) atomicExch(err, 1);
        __threadfence();
    }
    __syncthreads();
    return *failed == 0;
}

}  // namespace
