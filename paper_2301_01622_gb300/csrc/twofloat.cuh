// Numbers carried as an unevaluated sum h + l of two floats (h rounded to nearest,
// l the rounding error), for sums and differences that must not lose what FP64
// would keep.  GB300's FP64 pipe does two FMA per clock and SM; kernels that read
// FP32 and need a few more bits are several times faster on these.
// Sums by Knuth's two-sum, products by FMA; relative error about 2^-46.
#pragma once

namespace llb {

struct Two {
    float h = 0.0f, l = 0.0f;

    // a + b exactly
    __device__ __forceinline__ static Two sum(float a, float b) {
        const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
        return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
    }
    // a b exactly
    __device__ __forceinline__ static Two prod(float a, float b) {
        const float p = __fmul_rn(a, b);
        return {p, __fmaf_rn(a, b, -p)};
    }
    __device__ __forceinline__ void add(float a) {
        const Two s = sum(h, a);
        h = s.h;
        l = __fadd_rn(l, s.l);
    }
    __device__ __forceinline__ void add(const Two& o) {
        add(o.h);
        l = __fadd_rn(l, o.l);
    }
    // an infinite or NaN sum is h alone: its rounding error is not a number
    __device__ __forceinline__ double value() const { return isfinite(h) ? (double)h + (double)l : (double)h; }
    __device__ __forceinline__ Two shfl_down(int off) const {
        return {__shfl_down_sync(0xffffffffu, h, off), __shfl_down_sync(0xffffffffu, l, off)};
    }
};

// (h + l) / 3
__device__ __forceinline__ Two third(float h, float l) {
    constexpr float c = (float)(1.0 / 3.0), ce = (float)(1.0 / 3.0 - (double)c);
    Two p = Two::prod(h, c);
    p.l = __fmaf_rn(l, c, __fmaf_rn(h, ce, p.l));
    return p;
}

}  // namespace llb
