// Device arithmetic written for the latency of the Newton solves, with the bounds
// that tests/test_gpu_numerics.py checks.
#pragma once

#include <cuda_runtime.h>

namespace pt {

// 1/x rounded to nearest, for x in the middle of the FP32 range: the hardware's
// approximation and one residual correction (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34, 1990).
// Equal to __frcp_rn on every significand (tests/test_gpu_numerics.py checks all of
// them, at both signs); extreme exponents take __frcp_rn itself, whose call and
// branches cost about 240 dependent cycles in place of 80.
__device__ __forceinline__ float rcp_rn(float x) {
    if ((((unsigned)__float_as_int(x) >> 23 & 0xffu) - 64u) > 126u) return __frcp_rn(x);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
}
}  // namespace pt
