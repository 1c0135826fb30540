// FP64 reductions over the shifted moments (validation diagnostics of
// Sec. IV: droplet density <rho>_{rho > 0.5} of Figs. 2, 5, 7; total mass and
// momentum, which BGK collision and periodic streaming conserve).
//
// Pass 1: a fixed grid of blocks walks the nodes with a grid-stride loop,
// reduces in registers, then warp shuffles, then across the block's warps
// through shared memory, and writes one row of partials per block to a
// scratch array.  Pass 2: one block reduces the rows in a fixed order.  The
// result is deterministic for a given grid.  The sums of a thread and a warp are
// FP64 for FP64 data; for FP32 and 16-bit data they are sums of three floats,
// which are at least as accurate, and FP64 where those overflow.
#include <cuda_runtime.h>

#include <cfloat>
#include <mutex>
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"
#include "layout.cuh"
#include "storage.cuh"
#include "twofloat.cuh"

namespace llb {
namespace {

constexpr int kDiagThreads = 256;
constexpr int kRow = 9;  // sum d, sum jx, sum jy, sum jz, sum rho_in, n_in, min rho, nonfinite, sum rho1

struct Part {
    double v[kRow];
};

__device__ __forceinline__ void part_merge(Part& a, const Part& b) {
#pragma unroll
    for (int k = 0; k < 6; ++k) a.v[k] += b.v[k];
    a.v[6] = fmin(a.v[6], b.v[6]);
    a.v[7] = fmax(a.v[7], b.v[7]);
    a.v[8] += b.v[8];
}

__device__ __forceinline__ Part warp_reduce(Part p) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        Part o;
#pragma unroll
        for (int k = 0; k < kRow; ++k) o.v[k] = __shfl_down_sync(0xffffffffu, p.v[k], off);
        part_merge(p, o);
    }
    return p;
}

// Sums of one thread.  States and inputs of at most FP32 are summed in three floats
// (Sum3, twofloat.cuh): the FP64 form kept the FP64 pipe 79 % busy and took 106 us
// for the 92 MB of a 128^3 two-component state.
template <bool WIDE>
struct Sums;

template <>
struct Sums<true> {  // FP64 values
    double v[kRow];
    __device__ __forceinline__ Sums() {
        for (int k = 0; k < kRow; ++k) v[k] = 0.0;
        v[6] = DBL_MAX;
    }
    __device__ __forceinline__ void node(double d, double jx, double jy, double jz, double drop, bool two, bool finite) {
        const double rho = 1.0 + d;
        v[0] += d;
        v[1] += jx;
        v[2] += jy;
        v[3] += jz;
        if (drop > 0.5) {
            v[4] += drop;
            v[5] += 1.0;
        }
        v[6] = fmin(v[6], rho);
        if (!finite) v[7] = 1.0;
        if (two) v[8] += drop;
    }
    // one component from canonical rho (the sums are of the density as given)
    __device__ __forceinline__ void canonical(double rho, double jx, double jy, double jz, bool finite) {
        v[0] += rho - 1.0;
        v[1] += jx;
        v[2] += jy;
        v[3] += jz;
        if (rho > 0.5) {
            v[4] += rho;
            v[5] += 1.0;
        }
        v[6] = fmin(v[6], rho);
        if (!finite) v[7] = 1.0;
    }
    __device__ __forceinline__ bool row(Part& p) const {
        for (int k = 0; k < kRow; ++k) p.v[k] = v[k];
        p = warp_reduce(p);
        return true;
    }
};

template <>
struct Sums<false> {  // FP32 values
    Sum3 d, jx, jy, jz, in, all;  // in: sum of the droplet density (one component: of d) where it exceeds 0.5
    float dmin = INFINITY, rmin = INFINITY;
    unsigned n_in = 0, bad = 0;
    bool two = false;
    __device__ __forceinline__ void node(float dv, float x, float y, float z, float drop, bool two_, bool finite) {
        two = two_;
        d.add(dv);
        jx.add(x);
        jy.add(y);
        jz.add(z);
        // one component: rho = 1 + d > 0.5; its 1 is added with the count
        const float v = two_ ? drop : dv;
        if (v > (two_ ? 0.5f : -0.5f)) {
            in.add(v);
            ++n_in;
        }
        dmin = fminf(dmin, dv);
        if (!finite) bad = 1;
        if (two_) all.add(drop);
    }
    __device__ __forceinline__ void canonical(float rho, float x, float y, float z, bool finite) {
        const Two dv = Two::sum(rho, -1.0f);
        d.add(dv);
        jx.add(x);
        jy.add(y);
        jz.add(z);
        if (rho > 0.5f) {
            in.add(dv);
            ++n_in;
        }
        rmin = fminf(rmin, rho);
        if (!finite) bad = 1;
    }
    // Sums of the warp, in lane 0; false (in every lane) where one is not finite: a partial
    // sum beyond FP32's range, or data that is not finite.  They then have to be formed in FP64.
    __device__ __forceinline__ bool row(Part& p) {
        double n = 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            d.add(d.shfl_down(off));
            jx.add(jx.shfl_down(off));
            jy.add(jy.shfl_down(off));
            jz.add(jz.shfl_down(off));
            in.add(in.shfl_down(off));
            if (two) all.add(all.shfl_down(off));
            dmin = fminf(dmin, __shfl_down_sync(0xffffffffu, dmin, off));
            rmin = fminf(rmin, __shfl_down_sync(0xffffffffu, rmin, off));
            bad |= __shfl_down_sync(0xffffffffu, bad, off);
        }
        n = (double)__reduce_add_sync(0xffffffffu, n_in);
        p.v[0] = d.value();
        p.v[1] = jx.value();
        p.v[2] = jy.value();
        p.v[3] = jz.value();
        p.v[4] = in.value() + (two ? 0.0 : n);
        p.v[5] = n;
        p.v[6] = fmin(dmin == INFINITY ? DBL_MAX : 1.0 + (double)dmin, rmin == INFINITY ? DBL_MAX : (double)rmin);
        p.v[7] = (double)bad;
        p.v[8] = all.value();
        const bool held = isfinite(d.h) && isfinite(jx.h) && isfinite(jy.h) && isfinite(jz.h) && isfinite(in.h) && isfinite(all.h);
        return __shfl_sync(0xffffffffu, held, 0);
    }
};

// Row of partial sums of the block: (sum d, sum j, sum of the droplet density over
// nodes where it exceeds 0.5, their count, min rho, non-finite flag, sum rho1).
// The droplet density is rho for one component and rho1 for two (state
// rho1, d, j, A; rho2 = 1 + d - rho1 is recovered from the sums).
// walk(sums) adds the thread's nodes.
template <bool WIDE, class Walk>
__device__ __forceinline__ void write_row(Walk walk, bool two, double* __restrict__ row) {
    __shared__ double sh[kDiagThreads / 32][kRow];
    Part p;
    {
        Sums<WIDE> s;
        walk(s);
        if constexpr (!WIDE) s.two = two;  // a thread without nodes takes part in the same shuffles
        if (!s.row(p)) {
            Sums<true> w;
            walk(w);
            w.row(p);
        }
    }
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < kRow; ++k) sh[threadIdx.x >> 5][k] = p.v[k];
    __syncthreads();
    if (threadIdx.x < kRow) {
        const int k = threadIdx.x;
        double v = sh[0][k];
        for (int w = 1; w < kDiagThreads / 32; ++w) v = k == 6 ? fmin(v, sh[w][k]) : k == 7 ? fmax(v, sh[w][k]) : v + sh[w][k];
        row[k] = v;
    }
}

template <class T, int NC>
__global__ void __launch_bounds__(kDiagThreads) k_diag_partial(const T* __restrict__ m, Layout L,
                                                               double* __restrict__ rows) {
    constexpr bool WIDE = std::is_same<T, double>::value;
    using FM = FieldMap<T, 9 + NC>;
    const size_t N = (size_t)L.nx * L.ny * L.nz, F = L.fs;
    auto walk = [&](auto& s) {
        using V = typename std::conditional<std::is_same<decltype(s), Sums<true>&>::value, double, float>::type;
        for (size_t n = blockIdx.x * (size_t)kDiagThreads + threadIdx.x; n < N; n += (size_t)gridDim.x * kDiagThreads) {
            int x, y, z;
            if ((N >> 32) == 0) {  // 32-bit divisions when the box allows
                const unsigned q = (unsigned)n / (unsigned)L.nx;
                x = (int)((unsigned)n - q * (unsigned)L.nx);
                z = (int)(q / (unsigned)L.ny);
                y = (int)(q - (unsigned)z * (unsigned)L.ny);
            } else {
                x = (int)(n % L.nx);
                const size_t r = n / L.nx;
                y = (int)(r % L.ny);
                z = (int)(r / L.ny);
            }
            const size_t i = L.at(x, y, z);
            V v[9 + NC];
            bool finite = true;
#pragma unroll
            for (int f = 0; f < 9 + NC; ++f) {
                const T t = __ldg(m + FM::at(i, f, F));
                if constexpr (IsNarrow<T>::value) v[f] = cv_field<V>(t, f);
                else v[f] = (V)t;
                finite = finite && isfinite(v[f]);
            }
            s.node(v[NC - 1], v[NC], v[NC + 1], v[NC + 2], NC == 2 ? v[0] : V(1) + v[0], NC == 2, finite);
        }
    };
    write_row<WIDE>(walk, NC == 2, rows + (size_t)blockIdx.x * kRow);
}

// Sum of the rows, in a fixed order.
__global__ void __launch_bounds__(32 * kRow) k_diag_final(const double* __restrict__ rows, int nrows, size_t N,
                                                             int ncomp, llb_diag* __restrict__ out) {
    // 32 threads per column read the rows in order (coalesced), then a warp per column joins them
    __shared__ double part[kRow][33], sh[kRow];
    auto join = [](int k, double a, double b) { return k == 6 ? fmin(a, b) : k == 7 ? fmax(a, b) : a + b; };
    {
        const int k = threadIdx.x % kRow;
        double v = k == 6 ? DBL_MAX : 0.0;
#pragma unroll 8
        for (int i = threadIdx.x; i < nrows * kRow; i += 32 * kRow) v = join(k, v, rows[i]);
        part[k][threadIdx.x / kRow] = v;
    }
    __syncthreads();
    {
        const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
        double v = part[k][lane];
        for (int off = 16; off > 0; off >>= 1) v = join(k, v, __shfl_down_sync(0xffffffffu, v, off));
        if (lane == 0) sh[k] = v;
    }
    __syncthreads();
    Part p;
    if (threadIdx.x == 0)
        for (int q = 0; q < kRow; ++q) p.v[q] = sh[q];
    if (threadIdx.x == 0) {
        if (ncomp == 2) {
            out->mass[0] = p.v[8];
            out->mass[1] = (double)N + p.v[0] - p.v[8];
        } else {
            out->mass[0] = (double)N + p.v[0];
            out->mass[1] = 0.0;
        }
        out->momentum[0] = p.v[1];
        out->momentum[1] = p.v[2];
        out->momentum[2] = p.v[3];
        out->rho1_sum = p.v[4];
        out->n_in = (long long)p.v[5];
        out->rho1_avg = p.v[5] > 0.0 ? p.v[4] / p.v[5] : 0.0;
        const bool nonfinite = p.v[7] != 0.0;
        out->min_rho = nonfinite ? __longlong_as_double(0x7ff8000000000000ULL) : p.v[6];
        out->flags = (nonfinite ? LLB_FLAG_NONFINITE : 0) | (!nonfinite && p.v[6] <= 0.0 ? LLB_FLAG_NONPOSITIVE : 0);
        out->reserved = 0;
    }
}

}  // namespace

int diag_blocks(const llb_ctx& c) {
    const size_t want = (c.N + kDiagThreads - 1) / kDiagThreads;
    const size_t cap = (size_t)(c.num_sms > 0 ? c.num_sms : 148) * 4;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

cudaError_t launch_diagnostics(const llb_ctx& c, const void* mom, void* scratch, llb_diag* dev_out) {
    const int nb = diag_blocks(c);
    double* rows = static_cast<double*>(scratch);
    if (c.storage == LLB_F16S)
        k_diag_partial<__half, 1><<<nb, kDiagThreads, 0, c.stream>>>(static_cast<const __half*>(mom), c.lay, rows);
    else if (c.storage == LLB_BF16S)
        k_diag_partial<__nv_bfloat16, 1><<<nb, kDiagThreads, 0, c.stream>>>(static_cast<const __nv_bfloat16*>(mom),
                                                                             c.lay, rows);
    else if (c.ncomp == 2) {
        if (c.storage == LLB_F64)
            k_diag_partial<double, 2><<<nb, kDiagThreads, 0, c.stream>>>(static_cast<const double*>(mom), c.lay, rows);
        else
            k_diag_partial<float, 2><<<nb, kDiagThreads, 0, c.stream>>>(static_cast<const float*>(mom), c.lay, rows);
    } else {
        if (c.storage == LLB_F64)
            k_diag_partial<double, 1><<<nb, kDiagThreads, 0, c.stream>>>(static_cast<const double*>(mom), c.lay, rows);
        else
            k_diag_partial<float, 1><<<nb, kDiagThreads, 0, c.stream>>>(static_cast<const float*>(mom), c.lay, rows);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_diag_final<<<1, 32 * kRow, 0, c.stream>>>(rows, nb, c.N, c.ncomp, dev_out);
    return cudaGetLastError();
}

}  // namespace llb

// ---------------------------------------------------------------------------
// Diagnostics without allocation.
//
// Some callers cannot allocate device memory where they need the diagnostics:
// code running while a stream is being captured into a CUDA graph (a
// cudaMalloc there breaks the capture), allocator-owning frameworks and
// real-time loops that forbid allocation on the hot path, and embedders whose
// memory budget is fixed in advance.  For them the reduction below keeps its
// scratch (one row of partial sums per block plus the result) in a
// file-scope device array of fixed size, reserved when the library is loaded
// on a device and held until the process exits.
namespace llb {
namespace {

constexpr int kStaticRows = 4096;                       // partial-sum rows (one per block)
constexpr size_t kStaticNodesPerRow = (size_t)kDiagThreads * 64;
constexpr size_t kStaticMaxNodes = (size_t)kStaticRows * kStaticNodesPerRow;  // 67,108,864 nodes

struct StaticScratch {
    double rows[kStaticRows * kRow];
    llb_diag out;
};

// 288 KB of scratch per device.  Every call on a device reuses it: calls that
// overlap on the GPU (different streams, or different host threads without
// ordering) race on it.  Each call writes every row it later reads and the
// whole result, so no part of it has to be cleared between calls.
static __device__ __align__(256) StaticScratch g_diag_scratch;

// Partial sums of canonical one-component moments (rho, j, P), dense layout:
// block b reduces nodes [b * kStaticNodesPerRow, (b + 1) * kStaticNodesPerRow).
template <class T>
__global__ void __launch_bounds__(kDiagThreads) k_diag_partial_canonical(const T* __restrict__ m, size_t N,
                                                                         double* __restrict__ rows) {
    constexpr bool WIDE = std::is_same<T, double>::value;
    const size_t lo = (size_t)blockIdx.x * kStaticNodesPerRow;
    const size_t hi = lo + kStaticNodesPerRow < N ? lo + kStaticNodesPerRow : N;
    auto walk = [&](auto& s) {
        for (size_t i = lo + threadIdx.x; i < hi; i += kDiagThreads) {
            T v[10];
            bool finite = true;
#pragma unroll
            for (int f = 0; f < 10; ++f) {
                v[f] = __ldg(m + f * N + i);
                finite = finite && isfinite(v[f]);
            }
            s.canonical(v[0], v[1], v[2], v[3], finite);
        }
    };
    write_row<WIDE>(walk, false, rows + (size_t)blockIdx.x * kRow);
}

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
StaticScratch* g_static_ptr[kMaxDevices] = {};

}  // namespace
}  // namespace llb

extern "C" int llb_diagnostics_noalloc(const void* dev_m, int dtype, int nx, int ny, int nz, void* stream,
                                       llb_diag* host_out) {
    using namespace llb;
    if (!dev_m || !host_out || (dtype != LLB_F64 && dtype != LLB_F32) || nx < 1 || ny < 1 || nz < 1)
        return LLB_EINVAL;
    const size_t N = (size_t)nx * ny * nz;
    if (N > kStaticMaxNodes) return LLB_EINVAL;  // more nodes than the fixed scratch can reduce
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return LLB_ECUDA;
    }
    StaticScratch* scratch = nullptr;
    {
        // once per device, with that device current: the device address of the
        // array (its name in host code is only a host-side handle)
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ptr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_diag_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return LLB_ECUDA;
            }
            g_static_ptr[dev] = static_cast<StaticScratch*>(p);
        }
        scratch = g_static_ptr[dev];
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int nb = (int)((N + kStaticNodesPerRow - 1) / kStaticNodesPerRow);
    if (dtype == LLB_F64)
        k_diag_partial_canonical<double><<<nb, kDiagThreads, 0, s>>>(static_cast<const double*>(dev_m), N,
                                                                      scratch->rows);
    else
        k_diag_partial_canonical<float><<<nb, kDiagThreads, 0, s>>>(static_cast<const float*>(dev_m), N,
                                                                     scratch->rows);
    if (cudaGetLastError() != cudaSuccess) return LLB_ECUDA;
    k_diag_final<<<1, 32 * kRow, 0, s>>>(scratch->rows, nb, N, 1, &scratch->out);
    if (cudaGetLastError() != cudaSuccess) return LLB_ECUDA;
    if (cudaMemcpyAsync(host_out, &scratch->out, sizeof(llb_diag), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return LLB_ECUDA;
    }
    return LLB_OK;
}
