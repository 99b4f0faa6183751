// Single instructions that more than one kernel file uses.
#pragma once
#include <cuda_runtime.h>

namespace aok {

// 1 / x within 2^-23 of it; denormal arguments and results become zero.
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Atomic minimum without a return value (a reduction the SM does not wait for).
__device__ __forceinline__ void red_min_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("red.global.min.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

}  // namespace aok
