// Numbers carried as unevaluated sums of floats, for sums, differences and quotients that
// must not lose what FP64 would keep.  GB300's FP64 pipe does two FMA per clock and SM;
// kernels that read FP32 and need more bits are several times faster on these.  Sums by
// Knuth's two-sum, products by FMA: both exact while nothing overflows or, for products,
// underflows.
#pragma once

namespace llb {

// h + l, h rounded to nearest
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
};

// A sum carried as h + l + m: h and l stay a renormalised pair, m collects what their
// additions round off.  After n terms the error is at most about n^2 2^-75 of the largest
// partial sum; FP64 has n 2^-53, more than that up to n = 2^22.  Exact but for that while
// nothing overflows: check h, which stays infinite or NaN once a step of it was.
struct Sum3 {
    float h = 0.0f, l = 0.0f, m = 0.0f;

    __device__ __forceinline__ void add(float a) {
        const Two s = Two::sum(h, a), t = Two::sum(l, s.l);
        m = __fadd_rn(m, t.l);
        const Two r = Two::sum(s.h, t.h);
        h = r.h;
        l = r.l;
    }
    __device__ __forceinline__ void add(const Two& a) {
        add(a.h);
        add(a.l);
    }
    __device__ __forceinline__ void add(const Sum3& o) {
        add(o.h);
        add(o.l);
        m = __fadd_rn(m, o.m);
    }
    __device__ __forceinline__ double value() const { return (double)h + ((double)l + (double)m); }
    __device__ __forceinline__ Sum3 shfl_down(int off) const {
        return {__shfl_down_sync(0xffffffffu, h, off), __shfl_down_sync(0xffffffffu, l, off),
                __shfl_down_sync(0xffffffffu, m, off)};
    }
};

// a + b + c rounded once: b + c and a + (b + c) as exact pairs, their low parts added with
// rounding to odd, which keeps the last addition from rounding a second time (Boldo and
// Melquiond, "Emulation of a FMA and correctly rounded sums", 2008).
__device__ __forceinline__ float round_sum(float a, float b, float c) {
    const Two u = Two::sum(b, c), t = Two::sum(a, u.h), v = Two::sum(t.l, u.l);
    float odd = v.h;
    if (v.l != 0.0f && !(__float_as_uint(odd) & 1u))  // inexact and even: the neighbour on the side of the rest
        odd = __uint_as_float(__float_as_uint(odd) + ((v.l > 0.0f) == (odd > 0.0f) ? 1u : ~0u));
    return __fadd_rn(t.h, odd);
}

// (h + l) / 3 as three floats: quotients of the remainders, which are exact.  Error about 2^-70.
struct Third {
    float a, b, c;
    __device__ __forceinline__ Third(float h, float l) {
        constexpr float q = (float)(1.0 / 3.0);
        a = __fmul_rn(h, q);
        const Two r = Two::sum(__fmaf_rn(-3.0f, a, h), l);
        b = __fmul_rn(r.h, q);
        c = __fmul_rn(__fadd_rn(__fmaf_rn(-3.0f, b, r.h), r.l), q);
    }
};

}  // namespace llb
