// Conversions between the canonical moments of the ABI and the shifted
// device storage, and initialisation at local equilibrium.
//
// canonical (one component): rho, j_x, j_y, j_z, P_xx, P_yy, P_zz, P_xy, P_xz, P_yz
// shifted storage:           d = rho - 1, j, A = P - cs^2 rho I
// Equilibrium (second moment of Eq. (5)): P^eq = cs^2 rho I + rho u u, so
// A^eq = rho u u.  All conversions compute in FP64, or in several floats where both
// sides are at most FP32, and round the result to FP32 or FP64 once (16-bit states
// round that once more, to their format).
// Two components: canonical rho1, rho2, j, P; state rho1, d = rho1 + rho2 - 1,
// j, A (rho1 needs no shift: it lies in [0, rho]).
// Canonical buffers are dense; the shifted state follows the context's
// Layout (padded with periodic ghosts for the moment scheme), and every
// write to it also writes the node's ghost copies.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"
#include "layout.cuh"
#include "storage.cuh"
#include "twofloat.cuh"

namespace llb {
namespace {

template <class S>
__device__ __forceinline__ double rd(const void* p, size_t i) {
    return (double)static_cast<const S*>(p)[i];
}

__device__ __forceinline__ double rdt(const void* p, size_t i, int dt) {
    return dt == LLB_F64 ? rd<double>(p, i) : rd<float>(p, i);
}

__device__ __forceinline__ bool bad_rho(double r) { return !(r > 0.0) || !isfinite(r); }

// Node i of the dense canonical order (32-bit divisions when the box allows: they
// are per node and the 64-bit ones cost several times as much).
__device__ __forceinline__ void decode(const Layout& L, size_t i, int& x, int& y, int& z) {
    if ((i >> 32) == 0) {
        const unsigned j = (unsigned)i, r = j / (unsigned)L.nx;
        x = (int)(j - r * (unsigned)L.nx);
        z = (int)(r / (unsigned)L.ny);
        y = (int)(r - (unsigned)z * (unsigned)L.ny);
    } else {
        x = (int)(i % L.nx);
        const size_t r = i / L.nx;
        y = (int)(r % L.ny);
        z = (int)(r / L.ny);
    }
}

template <class T, int NF, class V>
__device__ __forceinline__ void put(T* __restrict__ st, const Layout& L, int x, int y, int z, const V* v) {
    T t[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f)
        if constexpr (NF == 10) t[f] = to_store<T>(v[f], f);
        else t[f] = (T)v[f];
    for_node_and_ghosts(L, x, y, [&](int gx, int gy) {
        const size_t j = L.at(gx, gy, z);
#pragma unroll
        for (int f = 0; f < NF; ++f) st[FieldMap<T, NF>::at(j, f, L.fs)] = t[f];
    });
}

// The maps between canonical and stored values, rounded once.  From FP32 to a
// state of at most FP32 they run on sums of floats (twofloat.cuh): in FP64 the two conversions
// of every value and the arithmetic kept the FP64 pipe 80 % busy and took three
// times as long as the memory needs.
template <class C, class T>
constexpr bool kTwoFloat = std::is_same<C, float>::value && !std::is_same<T, double>::value;

// Whether sums of floats hold the arithmetic of a node: its total density h and what is
// combined with it finite and far from both ends of the range.  An infinity or NaN has no
// low part, and very small values lose it; such nodes take the FP64 form.
__device__ __forceinline__ bool pairs_hold(float h, float a, float b, float c) {
    return h >= 0x1p-60f && h <= 0x1p60f && fabsf(a) <= 0x1p60f && fabsf(b) <= 0x1p60f && fabsf(c) <= 0x1p60f;
}

// P - rho / 3 and A + rho / 3 of a density rho = h + l, rounded once.  (In FP64 the product
// with 1/3 is rounded to 2^-54 of rho first; where P is close to rho / 3 that shows in A.)
__device__ __forceinline__ float less_third(float p, const Two& rho) {
    const Third t(rho.h, rho.l);
    const Two s = Two::sum(p, -t.a), x = Two::sum(s.l, -t.b);
    return round_sum(s.h, x.h, __fsub_rn(x.l, t.c));
}
__device__ __forceinline__ float plus_third(float a, const Two& rho) {
    const Third t(rho.h, rho.l);
    const Two s = Two::sum(a, t.a), x = Two::sum(s.l, t.b);
    return round_sum(s.h, x.h, __fadd_rn(x.l, t.c));
}

// State (rho1,) d, j, A of canonical (rho or rho1, rho2), j, P; returns whether the total
// density is not positive or, in FP64, not finite.
template <int NC>
__device__ __forceinline__ bool to_state(const double* v, double* o) {
    const double rho = NC == 2 ? v[0] + v[1] : v[0];
    if constexpr (NC == 2) o[0] = v[0];
    o[NC - 1] = rho - 1.0;
#pragma unroll
    for (int f = NC; f < 9 + NC; ++f) o[f] = f < NC + 3 || f >= NC + 6 ? v[f] : v[f] - kCs2 * rho;
    return bad_rho(rho);
}
template <int NC>
__device__ __forceinline__ bool to_state(const float* v, float* o) {
    Two rho{v[0], 0.0f};
    if constexpr (NC == 2) rho = Two::sum(v[0], v[1]);
    if (!pairs_hold(rho.h, v[NC + 3], v[NC + 4], v[NC + 5])) {
        double w[9 + NC], r[9 + NC];
#pragma unroll
        for (int f = 0; f < 9 + NC; ++f) w[f] = (double)v[f];
        const bool bad = to_state<NC>(w, r);
#pragma unroll
        for (int f = 0; f < 9 + NC; ++f) o[f] = (float)r[f];
        return bad;
    }
    if constexpr (NC == 2) o[0] = v[0];
    o[NC - 1] = NC == 2 ? round_sum(-1.0f, v[0], v[NC - 1]) : __fsub_rn(v[0], 1.0f);
#pragma unroll
    for (int f = NC; f < 9 + NC; ++f) o[f] = f < NC + 3 || f >= NC + 6 ? v[f] : less_third(v[f], rho);
    return false;
}

// The way back.
template <int NC>
__device__ __forceinline__ void to_canon(const double* v, double* o) {
    const double rho = 1.0 + v[NC - 1];
    o[0] = NC == 2 ? v[0] : rho;
    if constexpr (NC == 2) o[1] = rho - v[0];
#pragma unroll
    for (int f = NC; f < 9 + NC; ++f) o[f] = f < NC + 3 || f >= NC + 6 ? v[f] : v[f] + kCs2 * rho;
}
template <int NC>
__device__ __forceinline__ void to_canon(const float* v, float* o) {
    const Two rho = Two::sum(1.0f, v[NC - 1]);
    if (!pairs_hold(rho.h, v[NC + 3], v[NC + 4], v[NC + 5]) || (NC == 2 && !(fabsf(v[0]) <= 0x1p60f))) {
        double w[9 + NC], r[9 + NC];
#pragma unroll
        for (int f = 0; f < 9 + NC; ++f) w[f] = (double)v[f];
        to_canon<NC>(w, r);
#pragma unroll
        for (int f = 0; f < 9 + NC; ++f) o[f] = (float)r[f];
        return;
    }
    o[0] = NC == 2 ? v[0] : rho.h;
    if constexpr (NC == 2) o[1] = round_sum(1.0f, v[1], -v[0]);
#pragma unroll
    for (int f = NC; f < 9 + NC; ++f) o[f] = f < NC + 3 || f >= NC + 6 ? v[f] : plus_third(v[f], rho);
}

// Nodes i0 .. i1-1 of the dense canonical order (whole planes for a z-range).
// NC components; canonical rho (rho1, rho2), j, P; state (rho1,) d, j, A.
template <class C, class T, int NC>
__global__ void __launch_bounds__(256) k_canon_to_shifted(const C* __restrict__ canon, T* __restrict__ st, Layout L,
                                                          int* bad, size_t i0, size_t i1) {
    using V = typename std::conditional<kTwoFloat<C, T>, float, double>::type;
    constexpr int NF = 9 + NC;
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = i0 + blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < i1; i += (size_t)gridDim.x * blockDim.x) {
        V v[NF], o[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) v[f] = (V)__ldg(canon + f * N + i);
        // the total density must be positive; a colour density may dip slightly
        // below zero (the stepped colour-gradient field does so near interfaces)
        bool b = to_state<NC>(v, o);
#pragma unroll
        for (int f = 0; f < NF; ++f) b = b || !isfinite(v[f]);
        if (b && bad) atomicOr(bad, 1);
        int x, y, z;
        decode(L, i, x, y, z);
        put<T, NF>(st, L, x, y, z, o);
    }
}

template <class C, class T, int NC>
__global__ void __launch_bounds__(256) k_shifted_to_canon(const T* __restrict__ st, C* __restrict__ canon, Layout L,
                                                          size_t i0, size_t i1) {
    using V = typename std::conditional<kTwoFloat<C, T>, float, double>::type;
    constexpr int NF = 9 + NC;
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = i0 + blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < i1; i += (size_t)gridDim.x * blockDim.x) {
        int x, y, z;
        decode(L, i, x, y, z);
        const size_t j = L.at(x, y, z);
        V v[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const T t = __ldg(st + FieldMap<T, NF>::at(j, f, L.fs));
            if constexpr (IsNarrow<T>::value) v[f] = cv_field<V>(t, f);
            else v[f] = (V)t;
        }
        V o[NF];
        to_canon<NC>(v, o);
#pragma unroll
        for (int f = 0; f < NF; ++f) canon[f * N + i] = (C)o[f];
    }
}

template <class T>
__global__ void k_equilibrium(const void* __restrict__ rho_p, const void* __restrict__ u_p, int dt,
                              T* __restrict__ st, Layout L, int* bad) {
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        const double rho = rdt(rho_p, i, dt);
        const double ux = rdt(u_p, i, dt), uy = rdt(u_p, N + i, dt), uz = rdt(u_p, 2 * N + i, dt);
        if ((bad_rho(rho) || !isfinite(ux) || !isfinite(uy) || !isfinite(uz)) && bad) atomicOr(bad, 1);
        const double o[10] = {rho - 1.0, rho * ux, rho * uy, rho * uz, rho * ux * ux, rho * uy * uy,
                              rho * uz * uz, rho * ux * uy, rho * ux * uz, rho * uy * uz};
        int x, y, z;
        decode(L, i, x, y, z);
        put<T, 10>(st, L, x, y, z, o);
    }
}

template <class T>
__global__ void k_equilibrium2(const void* __restrict__ rho_p, const void* __restrict__ u_p, int dt,
                               T* __restrict__ st, Layout L, int* bad) {
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        const double r1 = rdt(rho_p, i, dt), r2 = rdt(rho_p, N + i, dt);
        const double rho = r1 + r2;
        const double ux = rdt(u_p, i, dt), uy = rdt(u_p, N + i, dt), uz = rdt(u_p, 2 * N + i, dt);
        if ((bad_rho(rho) || !isfinite(r1) || !isfinite(r2) || !isfinite(ux) || !isfinite(uy) || !isfinite(uz)) && bad)
            atomicOr(bad, 1);
        const double o[11] = {r1, rho - 1.0, rho * ux, rho * uy, rho * uz, rho * ux * ux, rho * uy * uy,
                              rho * uz * uz, rho * ux * uy, rho * ux * uz, rho * uy * uz};
        int x, y, z;
        decode(L, i, x, y, z);
        put<T, 11>(st, L, x, y, z, o);
    }
}

int grid_for(const llb_ctx& c, size_t nodes) {
    const size_t want = (nodes + 255) / 256;
    const size_t cap = (size_t)(c.num_sms > 0 ? c.num_sms : 148) * 8;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// fn(state element type, canonical element type, components)
template <class T>
struct Tag {
    using type = T;
};
template <class F>
void by_types(const llb_ctx& c, int cdt, F&& fn) {
    auto canon = [&](auto st, auto nc) {
        if (cdt == LLB_F64) fn(st, Tag<double>{}, nc);
        else fn(st, Tag<float>{}, nc);
    };
    using One = std::integral_constant<int, 1>;
    using Pair = std::integral_constant<int, 2>;
    if (c.storage == LLB_F16S) canon(Tag<__half>{}, One{});
    else if (c.storage == LLB_BF16S) canon(Tag<__nv_bfloat16>{}, One{});
    else if (c.ncomp == 2 && c.storage == LLB_F64) canon(Tag<double>{}, Pair{});
    else if (c.ncomp == 2) canon(Tag<float>{}, Pair{});
    else if (c.storage == LLB_F64) canon(Tag<double>{}, One{});
    else canon(Tag<float>{}, One{});
}

}  // namespace

cudaError_t launch_canonical_to_shifted_range(const llb_ctx& c, const void* canon, int cdt, void* st, int* bad, int zlo,
                                              int zhi, cudaStream_t s) {
    const size_t per = (size_t)c.nx * c.ny, i0 = per * zlo, i1 = per * zhi;
    by_types(c, cdt, [&](auto t, auto u, auto nc) {
        using T = typename decltype(t)::type;
        using C = typename decltype(u)::type;
        k_canon_to_shifted<C, T, decltype(nc)::value><<<grid_for(c, i1 - i0), 256, 0, s>>>(
            static_cast<const C*>(canon), static_cast<T*>(st), c.lay, bad, i0, i1);
    });
    return cudaGetLastError();
}

cudaError_t launch_shifted_to_canonical_range(const llb_ctx& c, const void* st, void* canon, int cdt, int zlo, int zhi,
                                              cudaStream_t s) {
    const size_t per = (size_t)c.nx * c.ny, i0 = per * zlo, i1 = per * zhi;
    by_types(c, cdt, [&](auto t, auto u, auto nc) {
        using T = typename decltype(t)::type;
        using C = typename decltype(u)::type;
        k_shifted_to_canon<C, T, decltype(nc)::value><<<grid_for(c, i1 - i0), 256, 0, s>>>(
            static_cast<const T*>(st), static_cast<C*>(canon), c.lay, i0, i1);
    });
    return cudaGetLastError();
}

cudaError_t launch_canonical_to_shifted(const llb_ctx& c, const void* canon, int cdt, void* st, int* bad) {
    return launch_canonical_to_shifted_range(c, canon, cdt, st, bad, 0, c.nz, c.stream);
}

cudaError_t launch_shifted_to_canonical(const llb_ctx& c, const void* st, void* canon, int cdt) {
    return launch_shifted_to_canonical_range(c, st, canon, cdt, 0, c.nz, c.stream);
}

cudaError_t launch_equilibrium(const llb_ctx& c, const void* rho, const void* u, int dt, void* st, int* bad) {
    if (c.storage == LLB_F16S) {
        k_equilibrium<__half><<<grid_for(c, c.N), 256, 0, c.stream>>>(rho, u, dt, static_cast<__half*>(st), c.lay, bad);
        return cudaGetLastError();
    }
    if (c.storage == LLB_BF16S) {
        k_equilibrium<__nv_bfloat16><<<grid_for(c, c.N), 256, 0, c.stream>>>(rho, u, dt, static_cast<__nv_bfloat16*>(st),
                                                                        c.lay, bad);
        return cudaGetLastError();
    }
    if (c.ncomp == 2) {
        if (c.storage == LLB_F64)
            k_equilibrium2<double><<<grid_for(c, c.N), 256, 0, c.stream>>>(rho, u, dt, static_cast<double*>(st), c.lay, bad);
        else
            k_equilibrium2<float><<<grid_for(c, c.N), 256, 0, c.stream>>>(rho, u, dt, static_cast<float*>(st), c.lay, bad);
        return cudaGetLastError();
    }
    if (c.storage == LLB_F64)
        k_equilibrium<double><<<grid_for(c, c.N), 256, 0, c.stream>>>(rho, u, dt, static_cast<double*>(st), c.lay, bad);
    else
        k_equilibrium<float><<<grid_for(c, c.N), 256, 0, c.stream>>>(rho, u, dt, static_cast<float*>(st), c.lay, bad);
    return cudaGetLastError();
}

}  // namespace llb
