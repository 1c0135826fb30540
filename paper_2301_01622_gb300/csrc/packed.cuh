// Arithmetic on two nodes at once: the packed FP32 instructions of sm_100, one
// issue slot for two results.  A float operand stands for both halves.
#pragma once

#include <cuda_runtime.h>

namespace llb {
namespace pk {

__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 mul(float a, float2 b) { return __fmul2_rn(make_float2(a, a), b); }
__device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 fma(float a, float2 b, float2 c) { return __ffma2_rn(make_float2(a, a), b, c); }
// exact: b * -1 is not rounded
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(make_float2(-1.0f, -1.0f), b, a); }

// Hardware approximations without the scaling that subnormal operands would need:
// 1 / (1 + s d) for a density of order one (within 1 ulp), and 1 / sqrt(x) for a
// normal x (within 2 ulp).
__device__ __forceinline__ float rcp1p(float s, float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaf(s, d, 1.0f)));
    return r;
}
__device__ __forceinline__ float2 rcp1p(float s, float2 d) { return make_float2(rcp1p(s, d.x), rcp1p(s, d.y)); }
__device__ __forceinline__ float rsqrt_fast(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

}  // namespace pk
}  // namespace llb
