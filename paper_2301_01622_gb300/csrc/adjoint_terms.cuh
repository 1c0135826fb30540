// Sums of the adjoint's dL/domega (adjoint.cu) over the nodes of a thread and a warp.
#pragma once

#include <cfloat>

#include "packed.cuh"
#include "twofloat.cuh"

namespace llb {

// dL/domega terms of a node, lam'_A : (j j / rho - A) with lam'_A = a, j j = b, 1 / rho = r,
// A = c, and their sums.  In FP64 these some 40 operations per node filled the FP64 pipe
// (two FMA per clock and SM; 79 % busy) and set the time of the adjoint step, 62 of 62 us
// on 128 x 96 x 64 D3Q19 FP32.  For an FP32 state they run on sums of floats
// (twofloat.cuh), every product and difference exact, which is more accurate than FP64;
// nodes whose terms leave the range where that holds run in FP64.  FP64 states keep FP64.
template <class T>
struct Wide;

template <>
struct Wide<double> {
    double v = 0.0;
    __device__ __forceinline__ void add_node(const double* a, const double* b, double r, const double* c) {
#pragma unroll
        for (int k = 0; k < 6; ++k) v += a[k] * (b[k] * r - c[k]);
    }
    // of the warp, in lane 0
    __device__ __forceinline__ double warp_sum() const {
        double s = v;
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        return s;
    }
};

// The largest |a| and the largest |b r| + |c| of a node's terms (or more than that).
struct TermSizes {
    float a, d;
    __device__ __forceinline__ TermSizes(const float* av, const float* b, float r, const float* c) {
        a = fabsf(av[0]);
        float bm = fabsf(b[0]), cm = fabsf(c[0]);
#pragma unroll
        for (int k = 1; k < 6; ++k) {
            a = fmaxf(a, fabsf(av[k]));
            bm = fmaxf(bm, fabsf(b[k]));
            cm = fmaxf(cm, fabsf(c[k]));
        }
        d = fmaf(bm, fabsf(r), cm);
    }
    // Whether sums of floats hold the terms as they are: nothing overflows, and what
    // underflows is below 2^-58 of a d.  No terms at all are held.
    __device__ __forceinline__ bool held() const {
        const float t = a * d;
        return (t >= 0x1p-88f && t <= 0x1p100f && d >= 0x1p-88f) || (a == 0.0f && d <= 0x1p100f) || (d == 0.0f && a <= 0x1p100f);
    }
};

// FP64 sum of this thread's nodes whose terms are not held (for FP32 states: few, so it lives
// in shared memory and costs no registers).
constexpr int kWideThreads = 128;
__device__ __forceinline__ double& wide_slot() {
    __shared__ double slot[kWideThreads];
    return slot[threadIdx.x];
}

// Two sums side by side, each as Sum3, of terms a (b r - c).
struct PairSums {
    float2 h = {0.0f, 0.0f}, l = {0.0f, 0.0f}, m = {0.0f, 0.0f};

    // x <- x + y rounded; returns what that rounds off
    static __device__ __forceinline__ float2 add_exact(float2& x, float2 y) {
        using namespace pk;
        const float2 s = add(x, y), t = sub(s, x), e = add(sub(x, sub(s, t)), sub(y, t));
        x = s;
        return e;
    }
    __device__ __forceinline__ void add_terms(float2 a, float2 b, float2 r, float2 c) {
        using namespace pk;
        // b r - c = s + t + tl exactly
        float2 s = mul(b, r);
        float2 t = fma(b, r, mul(-1.0f, s));
        const float2 sl = add_exact(s, mul(-1.0f, c)), tl = add_exact(t, sl);
        const float2 x = mul(a, s), y = mul(a, t);
        float2 u = fma(a, s, mul(-1.0f, x));
        const float2 yl = fma(a, t, mul(-1.0f, y));
        const float2 low = add(fma(a, tl, yl), add_exact(u, y));
        const float2 e = add_exact(l, add_exact(h, x));
        m = add(m, add(low, add(e, add_exact(l, u))));
    }
    // after a node's terms
    __device__ __forceinline__ void renormalise() { l = add_exact(h, l); }
    __device__ __forceinline__ Sum3 first() const { return {h.x, l.x, m.x}; }
    __device__ __forceinline__ Sum3 second() const { return {h.y, l.y, m.y}; }
};

// Sum of a node's terms that are not held as they are: scaled by powers of two to the
// middle of the range, or in FP64 where they are not finite.  A gradient has such nodes
// where its cotangents fade out (first pass of the 96^3 D3Q27 droplets, launched alone: 85 us
// a step, all of them in FP64 92).
struct NodeTerms {
    float a[6], b[6], c[6], r;
    __device__ __forceinline__ NodeTerms(const float* av, const float* bv, float rv, const float* cv) : r(rv) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            a[k] = av[k];
            b[k] = bv[k];
            c[k] = cv[k];
        }
    }
};
static __device__ __noinline__ double scaled_sum(NodeTerms n) {
    const float *const a = n.a, *const b = n.b, *const c = n.c, r = n.r;
    const TermSizes z(a, b, r, c);
    if (z.a > 0.0f && z.a <= FLT_MAX && z.d > 0.0f && z.d <= FLT_MAX) {
        const int ea = -ilogbf(z.a), ed = -ilogbf(z.d);
        // 2^ea and 2^ed as two factors each: up to 2^149
        const float a1 = ldexpf(1.0f, ea / 2), a2 = ldexpf(1.0f, ea - ea / 2);
        const float d1 = ldexpf(1.0f, ed / 2), d2 = ldexpf(1.0f, ed - ed / 2);
        PairSums v;
        for (int k = 0; k < 6; k += 2)
            v.add_terms(make_float2(a[k] * a1 * a2, a[k + 1] * a1 * a2), make_float2(b[k] * d1 * d2, b[k + 1] * d1 * d2),
                        make_float2(r, r), make_float2(c[k] * d1 * d2, c[k + 1] * d1 * d2));
        v.renormalise();
        Sum3 s = v.first();
        s.add(v.second());
        const double w = s.value();
        if (isfinite(w)) return ldexp(w, -ea - ed);
    }
    Wide<double> w;
    for (int k = 0; k < 6; ++k) w.v += (double)a[k] * ((double)b[k] * (double)r - (double)c[k]);
    return w.v;
}

template <>
struct Wide<float> {
    PairSums v;
    __device__ __forceinline__ Wide() { wide_slot() = 0.0; }
    // the terms in pairs: packed arithmetic, half the instructions
    __device__ __forceinline__ void add_node(const float* a, const float* b, float r, const float* c) {
        if (!TermSizes(a, b, r, c).held()) {
            wide_slot() += scaled_sum(NodeTerms(a, b, r, c));
            return;
        }
#pragma unroll
        for (int k = 0; k < 6; k += 2)
            v.add_terms(make_float2(a[k], a[k + 1]), make_float2(b[k], b[k + 1]), make_float2(r, r), make_float2(c[k], c[k + 1]));
        v.renormalise();
    }
    __device__ __forceinline__ double warp_sum() const {
        Sum3 s = v.first();
        s.add(v.second());
        for (int off = 16; off > 0; off >>= 1) s.add(s.shfl_down(off));
        double w = wide_slot();
        if (__any_sync(0xffffffffu, w != 0.0))
            for (int off = 16; off > 0; off >>= 1) w += __shfl_down_sync(0xffffffffu, w, off);
        return s.value() + w;
    }
};

}  // namespace llb
