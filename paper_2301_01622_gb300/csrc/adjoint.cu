// Hand-written adjoint of the one-component moment-only step.
//
// One step is m_new = S(C(m)) with
//   C (pointwise collision): (d, j, A) -> (d, j, A' = (1 - omega) A + omega j j / rho), rho = 1 + d
//   S (linear pull stencil): m_new(x) = sum_i e_i g_i(x - c_i),
//       g_i = r_i . m' = w_i [d + 3 c_i.j + 4.5 c_i c_i : A' - 1.5 tr A'],
//       e_i = (1, c_i, c_i c_i - cs^2 I) (the moments one unit of g_i carries).
// Its adjoint maps a cotangent lam_new of m_new to the cotangent of m:
//   lam'(y) = S^T lam_new (y) = sum_i r_i s_i,  s_i = e_i . lam_new(y + c_i)
//   lam(y)  = J_C(m(y))^T lam'(y)
// and accumulates dL/domega = sum_y lam'_A(y) : (j j / rho - A)(y).
// The state A is stored as six entries; a cotangent of an off-diagonal entry
// is the derivative with respect to that stored entry.
//
// Two components (A_h = 0, smooth normal |G|_eps): the state is (rho1, d, j,
// A) and a source node y emits g'_i (as above, with A' gaining
// ks n n, ks = A_s |G|_eps / 9, n = G / |G|_eps) and the colour population
//   h1'_i = (rho1 / rho)(w_i + g'_i) + e w_i (c_i.n) / |c_i|,  e = beta rho1 (rho - rho1) / rho,
// where G(y) = 3 sum_k w_k c_k phi(y + c_k), phi = 2 rho1 / rho - 1.  The
// adjoint runs in two passes: per node y, the cotangents of y's own fields
// and of G(y) (pull transposed, then the node's collision, perturbation and
// recolouring transposed); then per node z, the transposed gradient stencil
// lam_phi(z) = 3 sum_k w_k c_k . lam_G(z - c_k), added through phi(z) to
// lam_rho1(z) and lam_d(z).
//
// For two components the first pass (everything but the transposed gradient
// stencil) runs tiled by default (k_adjoint_cg_tiled, below); one component runs
// the march of the forward step for FP32 states (Adjoint, below) and the
// one-thread-per-node k_adjoint_step, a plain linear gather, for FP64.
//
// llb_adjoint runs the forward steps once, keeping the state every K steps
// (moments only), then walks the segments backwards: each segment is
// recomputed from its checkpoint with its K states kept, and the adjoint
// steps run through it in reverse (memory: ~N/K + K state copies).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "adjoint_terms.cuh"
#include "checked.cuh"
#include "internal.h"
#include "lattice.cuh"
#include "layout.cuh"
#include "moment_common.cuh"
#include "moment_pair.cuh"

namespace llb {
namespace {

constexpr int kAdjThreads = 128;

// Sum of the block's terms, added to its row (fixed order: warp shuffles, then the warps).
template <int NT, class T>
__device__ __forceinline__ void add_block_sum(const Wide<T>& part, double* __restrict__ row) {
    static_assert(NT <= kWideThreads, "a slot per thread");
    __shared__ double wsum[NT / 32];
    const double own = part.warp_sum();
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = own;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sacc = 0.0;
        for (int w = 0; w < NT / 32; ++w) sacc += wsum[w];
        *row += sacc;
    }
}

// The ten fields of node i of a one-component buffer (state or cotangent; the
// field order of FieldMap).
template <class T>
__device__ __forceinline__ void load10(const T* __restrict__ p, size_t i, size_t fs, T* v) {
#pragma unroll
    for (int f = 0; f < 10; ++f) v[f] = p[FieldMap<T, 10>::at(i, f, fs)];
}

// Adjoint of one step at source node y (one thread per node).  lam_new, m and
// lam share the context's Layout; neighbours are addressed with the periodic
// wrap (no ghost copies are needed in the cotangent arrays).
template <class L, class T>
__global__ void __launch_bounds__(kAdjThreads) k_adjoint_step(const T* __restrict__ lam_new, const T* __restrict__ m,
                                                              T* __restrict__ lam, Layout lay, T omega,
                                                              double* __restrict__ domega_rows) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    Wide<T> part;
    if (x < lay.nx) {
        // lam' = sum_i r_i (e_i . lam_new(y + c_i))
        T ld = T(0), lj[3] = {T(0), T(0), T(0)}, la[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
        for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cx = -1; cx <= 1; ++cx) {
                    if (!L::has(cx, cy, cz)) continue;
                    const size_t q = lay.at(wrap_idx(x + cx, lay.nx), wrap_idx(y + cy, lay.ny), wrap_idx(z + cz, lay.nz));
                    T v[10];
                    load10(lam_new, q, lay.fs, v);
                    const T cxx = T(cx * cx) - T(kCs2), cyy = T(cy * cy) - T(kCs2), czz = T(cz * cz) - T(kCs2);
                    // e_i . lam_new: the stored A entries carry (c_a c_b - cs^2 delta_ab)
                    const T si = v[0] + T(cx) * v[1] + T(cy) * v[2] + T(cz) * v[3] + cxx * v[4] + cyy * v[5] +
                                 czz * v[6] + T(cx * cy) * v[7] + T(cx * cz) * v[8] + T(cy * cz) * v[9];
                    const T ws = T(L::w(cx, cy, cz)) * si;
                    // r_i: dg/dd = w, dg/dj = 3 w c, dg/dA_aa = w (4.5 c_a^2 - 1.5), dg/dA_ab = 9 w c_a c_b
                    ld += ws;
                    lj[0] += T(3 * cx) * ws;
                    lj[1] += T(3 * cy) * ws;
                    lj[2] += T(3 * cz) * ws;
                    la[0] += (T(4.5 * cx * cx) - T(1.5)) * ws;
                    la[1] += (T(4.5 * cy * cy) - T(1.5)) * ws;
                    la[2] += (T(4.5 * cz * cz) - T(1.5)) * ws;
                    la[3] += T(9 * cx * cy) * ws;
                    la[4] += T(9 * cx * cz) * ws;
                    la[5] += T(9 * cy * cz) * ws;
                }
        // J_C^T at y
        const size_t i0 = lay.at(x, y, z);
        T s[10];
        load10(m, i0, lay.fs, s);
        const T rinv = T(1) / (T(1) + s[0]);
        const T jx = s[1], jy = s[2], jz = s[3];
        const T om = omega;
        // A'_aa = (1-w) A_aa + w j_a^2 / rho ; A'_ab = (1-w) A_ab + w j_a j_b / rho
        const T jj[6] = {jx * jx, jy * jy, jz * jz, jx * jy, jx * jz, jy * jz};
        T dsum = T(0);
        for (int k = 0; k < 6; ++k) dsum += la[k] * jj[k];
        T out[10];
        out[0] = ld - om * rinv * rinv * dsum;
        out[1] = lj[0] + om * rinv * (T(2) * jx * la[0] + jy * la[3] + jz * la[4]);
        out[2] = lj[1] + om * rinv * (T(2) * jy * la[1] + jx * la[3] + jz * la[5]);
        out[3] = lj[2] + om * rinv * (T(2) * jz * la[2] + jx * la[4] + jy * la[5]);
        for (int k = 0; k < 6; ++k) out[4 + k] = (T(1) - om) * la[k];
#pragma unroll
        for (int f = 0; f < 10; ++f) lam[FieldMap<T, 10>::at(i0, f, lay.fs)] = out[f];
        // dL/domega: lam'_A : (j j / rho - A)
        part.add_node(la, jj, rinv, s + 4);
    }
    add_block_sum<kAdjThreads>(part, domega_rows + ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x);
}

// Adjoint of one FP32 step on the march of the step itself (moment_pair.cuh).  A node
// publishes its s_i = e_i . lam_new, which has the form of the step's populations: a
// column with s = lam_d - tr lam_A / 3, j = -lam_j (the adjoint pulls from y + c_i) and
// a = lam_A.  The sums of the pull are the moments sum w_i s_i (1, -c, c c), from which
// r_i . s_i and J_C^T follow per node.  A thread holds two nodes; loading all ten fields
// of 19 neighbours per node, as k_adjoint_step does, kept the load pipe busy: 128 x 96 x
// 64 D3Q19 took 40.7 us a step, now about 31 (26.5 without the exact sums of dL/domega).
template <class L>
struct Adjoint {
    static constexpr bool kAdjoint = true;
    const float* m;
    float om;
    double* rows;

    struct Sum : PairSums {  // of the thread's two nodes (and wide_slot)
        __device__ __forceinline__ Sum() { wide_slot() = 0.0; }
    };

    // The sums of the pull are in units of the smallest weight w, up to 1 / w times their
    // moments: the columns carry a power of two that keeps them in the range of those.
    static constexpr float kDown = pk::Shells<L>::corners ? 0x1p-8f : 0x1p-6f;
    __device__ __forceinline__ pk::Col<float2> column(const float2* v) const {
        using namespace pk;
        Col<float2> c;
        c.jx = mul(-kDown, v[1]);
        c.jy = mul(-kDown, v[2]);
        c.jz = mul(-kDown, v[3]);
        c.xx = mul(kDown, v[4]);
        c.yy = mul(kDown, v[5]);
        c.zz = mul(kDown, v[6]);
        c.xy = mul(kDown, v[7]);
        c.xz = mul(kDown, v[8]);
        c.yz = mul(kDown, v[9]);
        c.s = col_s(c.xx, c.yy, c.zz, mul(kDown, v[0]));
        return c;
    }
    __device__ __forceinline__ void load(float* v, size_t e, size_t stride, size_t fs) const {
        if (!LLB_IN(e + 9 * stride, 10 * fs, kChkLoad)) return;
#pragma unroll
        for (int f = 0; f < 10; ++f) v[f] = load_dep(m + e + f * stride);
    }
    // r: sums of the pull in, cotangents of the two nodes (state a, b) out
    __device__ __forceinline__ void finish(float2* r, const float* a, const float* b, bool ok_lo, bool ok_hi,
                                           Sum& total) const {
        using namespace pk;
        constexpr double w = Shells<L>::w / kDown;
        constexpr float wh = (float)w, wl = (float)(w - (double)wh);
        float2 q[10];
#pragma unroll
        for (int f = 0; f < 10; ++f) q[f] = col_j(wh, wl, r[f]);
        float2 la[6];
        const float2 g15 = mul(-1.5f, q[0]);
#pragma unroll
        for (int f = 0; f < 3; ++f) la[f] = fma(4.5f, q[4 + f], g15);
#pragma unroll
        for (int f = 3; f < 6; ++f) la[f] = mul(9.0f, q[4 + f]);
        float2 s[10];
#pragma unroll
        for (int f = 0; f < 10; ++f) s[f] = make_float2(a[f], b[f]);
        const float2 one = make_float2(1.0f, 1.0f);
        const float2 r0 = rcp1p(1.0f, s[0]);
        const float2 rinv = fma(r0, sub(one, mul(r0, pk::add(one, s[0]))), r0);
        const float2 jx = s[1], jy = s[2], jz = s[3];
        const float2 jj[6] = {mul(jx, jx), mul(jy, jy), mul(jz, jz), mul(jx, jy), mul(jx, jz), mul(jy, jz)};
        // dL/domega: lam'_A : (j j / rho - A) of the nodes inside the box
        const bool ok[2] = {ok_lo, ok_hi};
        bool held = true;
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            float ta[6], tb[6], tc[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                ta[k] = n ? la[k].y : la[k].x;
                tb[k] = n ? jj[k].y : jj[k].x;
                tc[k] = n ? s[4 + k].y : s[4 + k].x;
            }
            held = held && TermSizes(ta, tb, n ? rinv.y : rinv.x, tc).held();
        }
        if (held) {
#pragma unroll
            for (int k = 0; k < 6; ++k)
                total.add_terms(make_float2(ok_lo ? la[k].x : 0.0f, ok_hi ? la[k].y : 0.0f), jj[k], rinv, s[4 + k]);
            total.renormalise();
        } else {
            // in FP64 and inline: the call of scaled_sum would spill registers (44 us a step, so 37,
            // launched alone)
            double w = 0.0;
#pragma unroll
            for (int n = 0; n < 2; ++n)
                if (ok[n])
                    for (int k = 0; k < 6; ++k)
                        w += (double)(n ? la[k].y : la[k].x) *
                             ((double)(n ? jj[k].y : jj[k].x) * (double)(n ? rinv.y : rinv.x) - (double)(n ? s[4 + k].y : s[4 + k].x));
            wide_slot() += w;
        }
        float2 dsum = mul(la[0], jj[0]);
#pragma unroll
        for (int k = 1; k < 6; ++k) dsum = fma(la[k], jj[k], dsum);
        const float2 o = mul(om, rinv);
        const float2 jx2 = pk::add(jx, jx), jy2 = pk::add(jy, jy), jz2 = pk::add(jz, jz);
        r[0] = sub(q[0], mul(mul(o, rinv), dsum));
        r[1] = fma(-3.0f, q[1], mul(o, fma(jx2, la[0], fma(jy, la[3], mul(jz, la[4])))));
        r[2] = fma(-3.0f, q[2], mul(o, fma(jy2, la[1], fma(jx, la[3], mul(jz, la[5])))));
        r[3] = fma(-3.0f, q[3], mul(o, fma(jz2, la[2], fma(jx, la[4], mul(jy, la[5])))));
#pragma unroll
        for (int k = 0; k < 6; ++k) r[4 + k] = mul(1.0f - om, la[k]);
    }
    __device__ __forceinline__ void end(const Sum& total) const {
        const double wide = wide_slot();
        Wide<float> part;  // (clears the slot)
        wide_slot() = wide;
        part.v = total;
        add_block_sum<mom::PairTile<L, mom::kPairH>::NT>(part, rows + blockIdx.x);
    }
};

template <class T>
struct CGAdjPar {
    T omega, beta, A_s, eps2;
};

__host__ __device__ constexpr double inv_len_c(int cx, int cy, int cz) {
    return (cx * cx + cy * cy + cz * cz) == 1 ? 1.0
         : (cx * cx + cy * cy + cz * cz) == 2 ? 0.70710678118654752440
         : (cx * cx + cy * cy + cz * cz) == 3 ? 0.57735026918962576451 : 0.0;
}

// Pass 1 of the two-component adjoint step at source node y: writes the
// cotangents of y's 11 fields (before the phase-field chain) to lam and of
// G(y) to lam_g (3 fields), and the block's dL/domega to domega_rows.
template <class L, class T>
__global__ void __launch_bounds__(kAdjThreads) k_adjoint_cg_local(const T* __restrict__ lam_new,
                                                                  const T* __restrict__ m, T* __restrict__ lam,
                                                                  T* __restrict__ lam_g, Layout lay, CGAdjPar<T> p,
                                                                  double* __restrict__ domega_rows) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    const size_t fs = lay.fs;
    Wide<T> part;
    if (x < lay.nx) {
        const size_t i0 = lay.at(x, y, z);
        T s[11];
#pragma unroll
        for (int f = 0; f < 11; ++f) s[f] = m[f * fs + i0];
        const T r1 = s[0], d = s[1], jx = s[2], jy = s[3], jz = s[4];
        const T* A = s + 5;  // xx, yy, zz, xy, xz, yz
        // G(y) from phi of the neighbours
        T G[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cx = -1; cx <= 1; ++cx) {
                    if (!L::has(cx, cy, cz) || (cx == 0 && cy == 0 && cz == 0)) continue;
                    const size_t q = lay.at(wrap_idx(x + cx, lay.nx), wrap_idx(y + cy, lay.ny), wrap_idx(z + cz, lay.nz));
                    const T ph = T(2) * m[q] / (T(1) + m[fs + q]) - T(1);
                    const T wp = T(3.0 * L::w(cx, cy, cz)) * ph;
                    G[0] += T(cx) * wp;
                    G[1] += T(cy) * wp;
                    G[2] += T(cz) * wp;
                }
        // forward quantities of the node
        const T rho = T(1) + d, rinv = T(1) / rho, om = p.omega;
        const T gn = sqrt(G[0] * G[0] + G[1] * G[1] + G[2] * G[2] + p.eps2);
        const T n[3] = {G[0] / gn, G[1] / gn, G[2] / gn};
        const T ks = p.A_s * gn * T(1.0 / 9.0);
        const T jj[6] = {jx * jx, jy * jy, jz * jz, jx * jy, jx * jz, jy * jz};
        const T nn[6] = {n[0] * n[0], n[1] * n[1], n[2] * n[2], n[0] * n[1], n[0] * n[2], n[1] * n[2]};
        T Ap[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) Ap[k] = (T(1) - om) * A[k] + om * jj[k] * rinv + ks * nn[k];
        const T s0 = d - T(1.5) * (Ap[0] + Ap[1] + Ap[2]);
        const T r1r = r1 * rinv;
        const T e = p.beta * r1 * (rho - r1) * rinv;
        // pull transposed: per direction, the cotangents of g'_i and h1'_i
        T ld = T(0), lj[3] = {T(0), T(0), T(0)}, la[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
        T l_r1r = T(0), l_e = T(0), ln[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cx = -1; cx <= 1; ++cx) {
                    if (!L::has(cx, cy, cz)) continue;
                    const size_t q = lay.at(wrap_idx(x + cx, lay.nx), wrap_idx(y + cy, lay.ny), wrap_idx(z + cz, lay.nz));
                    T v[11];
#pragma unroll
                    for (int f = 0; f < 11; ++f) v[f] = lam_new[f * fs + q];
                    const T cxx = T(cx * cx) - T(kCs2), cyy = T(cy * cy) - T(kCs2), czz = T(cz * cz) - T(kCs2);
                    const T si = v[1] + T(cx) * v[2] + T(cy) * v[3] + T(cz) * v[4] + cxx * v[5] + cyy * v[6] +
                                 czz * v[7] + T(cx * cy) * v[8] + T(cx * cz) * v[9] + T(cy * cz) * v[10];
                    const T ti = v[0];
                    const T w = T(L::w(cx, cy, cz));
                    T qd = s0;
                    if (cx) qd += T(4.5) * Ap[0];
                    if (cy) qd += T(4.5) * Ap[1];
                    if (cz) qd += T(4.5) * Ap[2];
                    if (cx * cy) qd += T(9 * cx * cy) * Ap[3];
                    if (cx * cz) qd += T(9 * cx * cz) * Ap[4];
                    if (cy * cz) qd += T(9 * cy * cz) * Ap[5];
                    const T gi = w * (qd + T(3 * cx) * jx + T(3 * cy) * jy + T(3 * cz) * jz);
                    l_r1r += ti * (w + gi);
                    if (cx || cy || cz) {
                        const T il = T(inv_len_c(cx, cy, cz));
                        const T cn = T(cx) * n[0] + T(cy) * n[1] + T(cz) * n[2];
                        l_e += ti * w * cn * il;
                        const T f = ti * e * w * il;
                        ln[0] += f * T(cx);
                        ln[1] += f * T(cy);
                        ln[2] += f * T(cz);
                    }
                    const T ws = w * (si + ti * r1r);
                    ld += ws;
                    lj[0] += T(3 * cx) * ws;
                    lj[1] += T(3 * cy) * ws;
                    lj[2] += T(3 * cz) * ws;
                    la[0] += (T(4.5 * cx * cx) - T(1.5)) * ws;
                    la[1] += (T(4.5 * cy * cy) - T(1.5)) * ws;
                    la[2] += (T(4.5 * cz * cz) - T(1.5)) * ws;
                    la[3] += T(9 * cx * cy) * ws;
                    la[4] += T(9 * cx * cz) * ws;
                    la[5] += T(9 * cy * cz) * ws;
                }
        // collision transposed: A' = (1 - w) A + w j j / rho + ks n n
        T l_rinv = T(0), l_ks = T(0);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            l_rinv += om * la[k] * jj[k];
            l_ks += la[k] * nn[k];
        }
        T out[11];
        out[2] = lj[0] + om * rinv * (T(2) * jx * la[0] + jy * la[3] + jz * la[4]);
        out[3] = lj[1] + om * rinv * (T(2) * jy * la[1] + jx * la[3] + jz * la[5]);
        out[4] = lj[2] + om * rinv * (T(2) * jz * la[2] + jx * la[4] + jy * la[5]);
#pragma unroll
        for (int k = 0; k < 6; ++k) out[5 + k] = (T(1) - om) * la[k];
        ln[0] += ks * (T(2) * n[0] * la[0] + n[1] * la[3] + n[2] * la[4]);
        ln[1] += ks * (T(2) * n[1] * la[1] + n[0] * la[3] + n[2] * la[5]);
        ln[2] += ks * (T(2) * n[2] * la[2] + n[0] * la[4] + n[1] * la[5]);
        // ks = A_s gn / 9, n = G / gn, gn = sqrt(|G|^2 + eps^2)
        T l_gn = p.A_s * T(1.0 / 9.0) * l_ks - (ln[0] * G[0] + ln[1] * G[1] + ln[2] * G[2]) / (gn * gn);
        T lg[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) lg[a] = ln[a] / gn + l_gn * G[a] / gn;
        // colour split: r1r = r1 / rho, e = beta (r1 - r1^2 / rho)
        l_rinv += l_r1r * r1 - l_e * p.beta * r1 * r1;
        out[0] = l_r1r * rinv + l_e * p.beta * (T(1) - T(2) * r1 * rinv);
        out[1] = ld - l_rinv * rinv * rinv;
#pragma unroll
        for (int f = 0; f < 11; ++f) lam[f * fs + i0] = out[f];
#pragma unroll
        for (int a = 0; a < 3; ++a) lam_g[a * fs + i0] = lg[a];
        part.add_node(la, jj, rinv, A);
    }
    add_block_sum<kAdjThreads>(part, domega_rows + ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x);
}

// Pass 2: the phase-field chain at node z.  G(y) = 3 sum_k w_k c_k phi(y + c_k)
// transposed gives lam_phi(z) = 3 sum_k w_k c_k . lam_G(z - c_k); phi = 2 rho1 / rho - 1.
//
// A thread walks kPhiPlanes planes of one (x, y).  The in-plane sums of a plane serve
// the three outputs around it, so it loads 9 neighbours per field and plane instead of
// 27, at addresses formed once.  96^3 D3Q27 FP32: 23 us before, 17.9 now (8 planes
// 20.6, too few warps for the latency of the loads; 1 plane 19.0).
constexpr int kPhiX = 32, kPhiY = 4, kPhiPlanes = 3;

template <class L, class T>
__global__ void __launch_bounds__(kPhiX * kPhiY) k_adjoint_cg_phi(const T* __restrict__ m, const T* __restrict__ lam_g,
                                                                  T* __restrict__ lam, Layout lay) {
    const int x = blockIdx.x * kPhiX + threadIdx.x, y = blockIdx.y * kPhiY + threadIdx.y;
    if (x >= lay.nx || y >= lay.ny) return;
    const int za = blockIdx.z * kPhiPlanes, zb = min(za + kPhiPlanes, lay.nz);
    const size_t fs = lay.fs, plane = (size_t)lay.px * lay.py;
    constexpr bool kC = L::has(1, 1, 1);
    constexpr T w1 = T(3.0 * L::w(1, 0, 0)), w2 = T(3.0 * L::w(1, 1, 0)), w3 = kC ? T(3.0 * L::w(1, 1, 1)) : T(0);
    size_t o[3][3];  // node (x + dx, y + dy) of plane 0 at [dy + 1][dx + 1]
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx)
            o[dy + 1][dx + 1] = LLB_CLAMP(lay.at(wrap_idx(x + dx, lay.nx), wrap_idx(y + dy, lay.ny), 0), fs, kChkLoad);
    // of one plane: c_z = 0 sum, c_z = +-1 sums of the x, y and of the z components, for
    // lam_phi(z) = 3 sum w c . lam_G(z - c): signs as if c pointed from z to its neighbour
    struct Sums { T d0, d1, s1; };
    auto plane_sums = [&](int z) {
        const size_t zo = (size_t)wrap_idx(z, lay.nz) * plane;
        T v[3][3][3];
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int i = 0; i < 3; ++i) v[f][j][i] = __ldg(lam_g + f * fs + o[j][i] + zo);
        const T ax = v[0][1][2] - v[0][1][0], ay = v[1][2][1] - v[1][0][1];
        const T xs = (v[0][2][2] - v[0][2][0]) + (v[0][0][2] - v[0][0][0]);
        const T ys = (v[1][2][2] - v[1][0][2]) + (v[1][2][0] - v[1][0][0]);
        const T za4 = (v[2][1][0] + v[2][1][2]) + (v[2][0][1] + v[2][2][1]);
        Sums r;
        r.d0 = w1 * (ax + ay) + w2 * (xs + ys);
        r.d1 = w2 * (ax + ay);
        r.s1 = w1 * v[2][1][1] + w2 * za4;
        if (kC) {
            r.d1 += w3 * (xs + ys);
            r.s1 += w3 * ((v[2][0][0] + v[2][0][2]) + (v[2][2][0] + v[2][2][2]));
        }
        return r;
    };
    Sums lo = plane_sums(za - 1), mid = plane_sums(za);
    for (int z = za; z < zb; ++z) {
        const Sums hi = plane_sums(z + 1);
        // the neighbour at z - c carries -c of the sums above
        const T lphi = -(mid.d0 + (lo.d1 + hi.d1) + (hi.s1 - lo.s1));
        const size_t i0 = LLB_CLAMP(o[1][1] + (size_t)z * plane, fs, kChkStore);
        const T rinv = T(1) / (T(1) + m[fs + i0]);
        lam[i0] += lphi * T(2) * rinv;
        lam[fs + i0] -= lphi * T(2) * m[i0] * rinv * rinv;
        lo = mid;
        mid = hi;
    }
}

// ---------------------------------------------------------------------------
// Tiled pass 1 of the two-component adjoint (the default).  Receiver y needs,
// for every direction c, s_c(y + c) = e_c . lam_new(y + c) and
// t(y + c) = lam_new_rho1(y + c), and phi(y + c) for G(y).  Instead of loading
// the 11 cotangent fields of each of its Q neighbours (k_adjoint_cg_local), a
// persistent CTA marches a BX x BY tile through z: for each plane, every node
// of the tile plus a one-node halo computes its Q projections once and
// publishes them, with t and phi, into a ring of three planes in shared
// memory; each receiver of the middle plane then reads two values per
// direction.  Two barriers per plane (published; ring slot free again).
//
// Everything the receiver needs is linear in the moments over the directions of s
// and t (sum w s (1, c, c c) and the same of t), in sum w c t / |c| and in G.  It forms
// those plane by plane from sums over directions of one weight and only then applies
// its own fields, where it evaluated the node's populations and their cotangents
// direction by direction (2160 instructions per node on D3Q27).  Twelve warps per SM
// (the ring) leave the loads exposed, so each plane is loaded one plane ahead: 96^3
// D3Q27 FP32 91 us a step before, 71 so (95 without the loads ahead), about 82 with the
// exact sums of dL/domega.
template <class L, class T, int BX, int BY>
struct AdjTile {
    static constexpr int NT = BX * BY, HX = BX + 2, HY = BY + 2, HN = HX * HY;
    static constexpr int NF = L::Q + 2;  // Q projections, (t, phi) of a node side by side
    static_assert(HN % 2 == 0, "aligned pairs");
    static constexpr int SLOT = NF * HN;  // elements of one plane of the ring
    static constexpr size_t smem_bytes = 3 * (size_t)SLOT * sizeof(T);
    static constexpr int MINB = sizeof(T) == 4 ? 3 : 1;  // CTAs per SM the register budget targets
    static_assert(NT % 32 == 0, "whole warps");
};
constexpr int kAdjBX = 32, kAdjBY = 4;

template <class T>
struct alignas(2 * sizeof(T)) Pair2 {
    T t, phi;
};

// Values of a field at the nine nodes of a plane around a node: at the node, at
// x +- 1, at y +- 1 and at the diagonal ones (1,1) (-1,-1) (1,-1) (-1,1).
template <class T>
struct Nine {
    T o, xp, xm, yp, ym, pp, mm, pm, mp;
};

// Sums over a plane's directions with weights wo (own column), wa (axes), wd (diagonals).
template <bool DIAG, class T>
__device__ __forceinline__ pk::PlaneSum<T> weighted(const Nine<T>& v, T wo, T wa, T wd) {
    pk::PlaneSum<T> q;
    const T sx = v.xp + v.xm, sy = v.yp + v.ym;
    q.g = wo * v.o + wa * (sx + sy);
    q.jx = wa * (v.xp - v.xm);
    q.jy = wa * (v.yp - v.ym);
    q.xx = wa * sx;
    q.yy = wa * sy;
    q.xy = T(0);
    if (DIAG) {
        const T sp = v.pp + v.mm, sm = v.pm + v.mp, dp = v.pp - v.mm, dm = v.pm - v.mp, sd = sp + sm;
        q.g += wd * sd;
        q.jx += wd * (dp + dm);
        q.jy += wd * (dp - dm);
        q.xx += wd * sd;
        q.yy += wd * sd;
        q.xy = wd * (sp - sm);
    }
    return q;
}

// sum w (1; c; c c) over all directions from the three planes (c_z = -1, 0, 1).
template <class T>
struct Sums10 {
    T g, j[3], a[6];
    __device__ __forceinline__ Sums10(const pk::PlaneSum<T>& m, const pk::PlaneSum<T>& z, const pk::PlaneSum<T>& p) {
        a[2] = p.g + m.g;
        g = z.g + a[2];
        j[0] = z.jx + (p.jx + m.jx);
        j[1] = z.jy + (p.jy + m.jy);
        j[2] = p.g - m.g;
        a[0] = z.xx + (p.xx + m.xx);
        a[1] = z.yy + (p.yy + m.yy);
        a[3] = z.xy + (p.xy + m.xy);
        a[4] = p.jx - m.jx;
        a[5] = p.jy - m.jy;
    }
};

// Index of direction (cx, cy, cz) in the lattice, enumerated over cz, cy, cx.
template <class L>
__host__ __device__ constexpr int dir_index(int cx, int cy, int cz) {
    int k = 0;
    for (int z = -1; z <= 1; ++z)
        for (int y = -1; y <= 1; ++y)
            for (int x = -1; x <= 1; ++x) {
                if (!L::has(x, y, z)) continue;
                if (x == cx && y == cy && z == cz) return k;
                ++k;
            }
    return -1;
}

// What a region node publishes from: its 11 cotangents, rho1 and d.
template <class T>
struct AdjNode {
    T v[11], r1, d;
    __device__ __forceinline__ void load(const T* __restrict__ lam_new, const T* __restrict__ m, size_t i, size_t fs) {
        if (!LLB_IN(i, fs, kChkLoad)) return;
#pragma unroll
        for (int f = 0; f < 11; ++f) v[f] = __ldg(lam_new + f * fs + i);
        r1 = __ldg(m + i);
        d = __ldg(m + fs + i);
    }
};

// Publish node j of the tile-plus-halo region into slot S.
template <class L, class T, int HN>
__device__ __forceinline__ void adj_publish(const AdjNode<T>& a, int j, T* __restrict__ S) {
    if (!LLB_IN(j, HN, kChkPublish)) return;
    const T* const v = a.v;
    *reinterpret_cast<Pair2<T>*>(S + L::Q * HN + 2 * j) = Pair2<T>{v[0], T(2) * a.r1 / (T(1) + a.d) - T(1)};
    // s(+-c) = even +- odd, even = v1 + (cc - cs^2 I) : vP, odd = c . vj
    const T ev0 = v[1] - T(kCs2) * (v[5] + v[6] + v[7]);
    S[dir_index<L>(0, 0, 0) * HN + j] = ev0;
#pragma unroll
    for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
        for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
            for (int cx = -1; cx <= 1; ++cx) {
                const bool lead = cx > 0 || (cx == 0 && (cy > 0 || (cy == 0 && cz > 0)));
                if (!lead || !L::has(cx, cy, cz)) continue;
                T ev = ev0;
                if (cx) ev += v[5];
                if (cy) ev += v[6];
                if (cz) ev += v[7];
                if (cx * cy) ev += T(cx * cy) * v[8];
                if (cx * cz) ev += T(cx * cz) * v[9];
                if (cy * cz) ev += T(cy * cz) * v[10];
                T od = T(0);
                if (cx) od += T(cx) * v[2];
                if (cy) od += T(cy) * v[3];
                if (cz) od += T(cz) * v[4];
                S[dir_index<L>(cx, cy, cz) * HN + j] = ev + od;
                S[dir_index<L>(-cx, -cy, -cz) * HN + j] = ev - od;
            }
}

// Receiver y (node n of the region, own 11 fields in s): the direct kernel's
// arithmetic with the neighbour quantities read from the ring planes Sm, S0, Sp
// (planes z - 1, z, z + 1).  Writes lam(y), lam_g(y); adds y's dL/domega term to part.
template <class L, class T, int HX, int HN>
__device__ __forceinline__ void adj_receive(Wide<T>& part, const T* __restrict__ Sm, const T* __restrict__ S0,
                                            const T* __restrict__ Sp, int n, const T* s, const CGAdjPar<T>& p,
                                            T* __restrict__ lam, T* __restrict__ lam_g, size_t i0, size_t fs) {
    if (!LLB_IN(n - HX - 1, HN, kChkGather) || !LLB_IN(n + HX + 1, HN, kChkGather) || !LLB_IN(i0, fs, kChkStore))
        return;
    constexpr int Q = L::Q;
    const T r1 = s[0], d = s[1], jx = s[2], jy = s[3], jz = s[4];
    const T* A = s + 5;  // xx, yy, zz, xy, xz, yz
    constexpr bool kC = L::has(1, 1, 1);
    constexpr T w0 = T(L::w(0, 0, 0)), w1 = T(L::w(1, 0, 0)), w2 = T(L::w(1, 1, 0)), w3 = kC ? T(L::w(1, 1, 1)) : T(0);
    // moments of s: the projection along c of the neighbour at y + c
    auto s9 = [&](const T* P, auto czc) {
        constexpr int cz = decltype(czc)::value;
        auto at = [&](auto cxc, auto cyc) -> T {
            constexpr int cx = decltype(cxc)::value, cy = decltype(cyc)::value;
            if constexpr (L::has(cx, cy, cz)) return P[dir_index<L>(cx, cy, cz) * HN + n + cy * HX + cx];
            else return T(0);
        };
        constexpr std::integral_constant<int, 0> o{};
        constexpr std::integral_constant<int, 1> p1{};
        constexpr std::integral_constant<int, -1> m1{};
        return Nine<T>{at(o, o), at(p1, o), at(m1, o), at(o, p1), at(o, m1), at(p1, p1), at(m1, m1), at(p1, m1), at(m1, p1)};
    };
    const Sums10<T> S(weighted<kC>(s9(Sm, std::integral_constant<int, -1>{}), w1, w2, w3),
                      weighted<true>(s9(S0, std::integral_constant<int, 0>{}), w0, w1, w2),
                      weighted<kC>(s9(Sp, std::integral_constant<int, 1>{}), w1, w2, w3));
    // moments of t, K = sum w c t / |c| and G = 3 sum w c phi
    auto t9 = [&](const T* P, Nine<T>& t, Nine<T>& f) {
        const Pair2<T>* const q = reinterpret_cast<const Pair2<T>*>(P + Q * HN) + n;
        auto rd = [&](int off, T& a, T& b) {
            const Pair2<T> v = q[off];
            a = v.t;
            b = v.phi;
        };
        rd(0, t.o, f.o);
        rd(1, t.xp, f.xp);
        rd(-1, t.xm, f.xm);
        rd(HX, t.yp, f.yp);
        rd(-HX, t.ym, f.ym);
        rd(HX + 1, t.pp, f.pp);
        rd(-HX - 1, t.mm, f.mm);
        rd(1 - HX, t.pm, f.pm);
        rd(HX - 1, t.mp, f.mp);
    };
    constexpr T k1 = T(L::w(1, 0, 0)), k2 = T(L::w(1, 1, 0) * inv_len_c(1, 1, 0)),
                k3 = kC ? T(L::w(1, 1, 1) * inv_len_c(1, 1, 1)) : T(0);
    T K[3], G[3];
    Nine<T> tv, fv;
    t9(Sm, tv, fv);
    const pk::PlaneSum<T> tm = weighted<kC>(tv, w1, w2, w3), fm = weighted<kC>(fv, w1, w2, w3),
                          km = weighted<kC>(tv, k1, k2, k3);
    t9(Sp, tv, fv);
    const pk::PlaneSum<T> tp = weighted<kC>(tv, w1, w2, w3), fp = weighted<kC>(fv, w1, w2, w3),
                          kp = weighted<kC>(tv, k1, k2, k3);
    t9(S0, tv, fv);
    const pk::PlaneSum<T> tz = weighted<true>(tv, w0, w1, w2), fz = weighted<true>(fv, T(0), w1, w2),
                          kz = weighted<true>(tv, T(0), k1, k2);
    const Sums10<T> M(tm, tz, tp);
    K[0] = kz.jx + (kp.jx + km.jx);
    K[1] = kz.jy + (kp.jy + km.jy);
    K[2] = kp.g - km.g;
    G[0] = T(3) * (fz.jx + (fp.jx + fm.jx));
    G[1] = T(3) * (fz.jy + (fp.jy + fm.jy));
    G[2] = T(3) * (fp.g - fm.g);
    const T rho = T(1) + d, rinv = T(1) / rho, om = p.omega;
    const T gn = sqrt(G[0] * G[0] + G[1] * G[1] + G[2] * G[2] + p.eps2);
    const T ign = T(1) / gn;
    const T nv[3] = {G[0] * ign, G[1] * ign, G[2] * ign};
    const T ks = p.A_s * gn * T(1.0 / 9.0);
    const T jj[6] = {jx * jx, jy * jy, jz * jz, jx * jy, jx * jz, jy * jz};
    const T nn[6] = {nv[0] * nv[0], nv[1] * nv[1], nv[2] * nv[2], nv[0] * nv[1], nv[0] * nv[2], nv[1] * nv[2]};
    T Ap[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) Ap[k] = (T(1) - om) * A[k] + om * jj[k] * rinv + ks * nn[k];
    const T s0 = d - T(1.5) * (Ap[0] + Ap[1] + Ap[2]);
    const T r1r = r1 * rinv;
    const T e = p.beta * r1 * (rho - r1) * rinv;
    // g'_i + w_i = w_i (1 + s0 + 3 c.j + 4.5 c c : A') summed over the directions with t
    T l_r1r = (T(1) + s0) * M.g + T(3) * (jx * M.j[0] + jy * M.j[1] + jz * M.j[2]);
    T l_e = T(0), ln[3], lj[3], la[6];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        l_r1r += T(4.5) * Ap[a] * M.a[a] + T(9) * Ap[3 + a] * M.a[3 + a];
        l_e += nv[a] * K[a];
        ln[a] = e * K[a];
    }
    const T ld = S.g + r1r * M.g;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lj[a] = T(3) * (S.j[a] + r1r * M.j[a]);
        la[a] = T(4.5) * (S.a[a] + r1r * M.a[a]) - T(1.5) * ld;
        la[3 + a] = T(9) * (S.a[3 + a] + r1r * M.a[3 + a]);
    }
    T l_rinv = T(0), l_ks = T(0);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        l_rinv += om * la[k] * jj[k];
        l_ks += la[k] * nn[k];
    }
    T out[11];
    out[2] = lj[0] + om * rinv * (T(2) * jx * la[0] + jy * la[3] + jz * la[4]);
    out[3] = lj[1] + om * rinv * (T(2) * jy * la[1] + jx * la[3] + jz * la[5]);
    out[4] = lj[2] + om * rinv * (T(2) * jz * la[2] + jx * la[4] + jy * la[5]);
#pragma unroll
    for (int k = 0; k < 6; ++k) out[5 + k] = (T(1) - om) * la[k];
    ln[0] += ks * (T(2) * nv[0] * la[0] + nv[1] * la[3] + nv[2] * la[4]);
    ln[1] += ks * (T(2) * nv[1] * la[1] + nv[0] * la[3] + nv[2] * la[5]);
    ln[2] += ks * (T(2) * nv[2] * la[2] + nv[0] * la[4] + nv[1] * la[5]);
    const T l_gn = p.A_s * T(1.0 / 9.0) * l_ks - (ln[0] * nv[0] + ln[1] * nv[1] + ln[2] * nv[2]) * ign;
    l_rinv += l_r1r * r1 - l_e * p.beta * r1 * r1;
    out[0] = l_r1r * rinv + l_e * p.beta * (T(1) - T(2) * r1 * rinv);
    out[1] = ld - l_rinv * rinv * rinv;
#pragma unroll
    for (int f = 0; f < 11; ++f) lam[f * fs + i0] = out[f];
#pragma unroll
    for (int a = 0; a < 3; ++a) lam_g[a * fs + i0] = ln[a] * ign + l_gn * nv[a];
    part.add_node(la, jj, rinv, A);
}

template <class L, class T, int BX, int BY>
__global__ void __launch_bounds__(BX * BY, (AdjTile<L, T, BX, BY>::MINB))
    k_adjoint_cg_tiled(const T* __restrict__ lam_new, const T* __restrict__ m, T* __restrict__ lam,
                       T* __restrict__ lam_g, Layout lay, CGAdjPar<T> p, mom::Sched sc,
                       double* __restrict__ domega_rows) {
    using C = AdjTile<L, T, BX, BY>;
    constexpr int NT = C::NT, HX = C::HX, HN = C::HN, SLOT = C::SLOT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* const ring = reinterpret_cast<T*>(smem_raw);
    const int nx = lay.nx, ny = lay.ny, nz = lay.nz;
    const size_t fs = lay.fs, plane = (size_t)lay.px * lay.py;
    const int t = threadIdx.x, tx = t % BX, ty = t / BX;
    const int n_own = (ty + 1) * HX + (tx + 1);
    Wide<T> part;

    for (int it = blockIdx.x; it < sc.nitems; it += gridDim.x) {
        int x0, y0, za, zb;  // receivers of planes za .. zb-1 of the tile at (x0, y0)
        sc.item(it, BX, BY, nz, x0, y0, za, zb);
        // region nodes of this thread: j = t and j = t + NT (if inside the tile plus halo)
        const int j1 = t + NT;
        const size_t off0 = lay.at(mom::pmod(x0 - 1 + t % HX, nx), mom::pmod(y0 - 1 + t / HX, ny), 0);
        const size_t off1 = j1 < HN ? lay.at(mom::pmod(x0 - 1 + j1 % HX, nx), mom::pmod(y0 - 1 + j1 / HX, ny), 0) : 0;
        const int ox = x0 + tx, oy = y0 + ty;
        const bool ok = ox < nx && oy < ny;
        const size_t own = ok ? lay.at(ox, oy, 0) : 0;
        auto slot = [&](int q) { return ring + (size_t)((q - za + 1) % 3) * SLOT; };  // q >= za - 1
        // a plane is loaded while the one before it is received
        AdjNode<T> a0, a1;
        auto load = [&](int q) {
            const size_t zo = (size_t)mom::pmod(q, nz) * plane;
            a0.load(lam_new, m, off0 + zo, fs);
            if (j1 < HN) a1.load(lam_new, m, off1 + zo, fs);
        };
        auto publish = [&](int q) {
            T* S = slot(q);
            adj_publish<L, T, HN>(a0, t, S);
            if (j1 < HN) adj_publish<L, T, HN>(a1, j1, S);
        };
        load(za - 1);
        publish(za - 1);
        load(za);
        publish(za);
        load(za + 1);
        for (int q = za; q < zb; ++q) {  // receivers of plane q
            publish(q + 1);
            if (q + 2 <= zb) load(q + 2);
            T sv[11];
            const size_t iy = own + (size_t)mom::pmod(q, nz) * plane;
            if (ok && LLB_IN(iy, fs, kChkLoad)) {
#pragma unroll
                for (int f = 0; f < 11; ++f) sv[f] = m[f * fs + iy];
            }
            __syncthreads();  // planes q - 1, q, q + 1 published
            if (ok) adj_receive<L, T, HX, HN>(part, slot(q - 1), slot(q), slot(q + 1), n_own, sv, p, lam, lam_g, iy, fs);
            __syncthreads();  // the slot of plane q - 1 may be refilled
        }
    }
    add_block_sum<NT>(part, domega_rows + blockIdx.x);
}

// acc += sum of rows (one block, fixed order).
__global__ void k_sum_rows(const double* __restrict__ rows, size_t n, double* __restrict__ acc) {
    __shared__ double sh[256];
    double s = 0.0;
    for (size_t i = threadIdx.x; i < n; i += 256) s += rows[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *acc += sh[0];
}

// Cotangents: canonical (rho, j, P) <-> shifted (d, j, A).  The forward maps are
// d = rho - 1, A_aa = P_aa - cs^2 rho, A_ab = P_ab and back rho = 1 + d,
// P_aa = A_aa + cs^2 (1 + d); the cotangent maps are their transposes.
template <class T>
__global__ void k_cot_canon_to_shifted(const void* __restrict__ g, int dt, T* __restrict__ lam, Layout L) {
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        double v[10];
        for (int f = 0; f < 10; ++f)
            v[f] = dt == LLB_F64 ? static_cast<const double*>(g)[f * N + i] : (double)static_cast<const float*>(g)[f * N + i];
        const int x = (int)(i % L.nx);
        const size_t r = i / L.nx;
        const size_t j = L.at(x, (int)(r % L.ny), (int)(r / L.ny));
        lam[FieldMap<T, 10>::at(j, 0, L.fs)] = (T)(v[0] + kCs2 * (v[4] + v[5] + v[6]));
        for (int f = 1; f < 10; ++f) lam[FieldMap<T, 10>::at(j, f, L.fs)] = (T)v[f];
    }
}

template <class T>
__global__ void k_cot_shifted_to_canon(const T* __restrict__ lam, void* __restrict__ g, int dt, Layout L) {
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % L.nx);
        const size_t r = i / L.nx;
        const size_t j = L.at(x, (int)(r % L.ny), (int)(r / L.ny));
        double v[10];
        for (int f = 0; f < 10; ++f) v[f] = (double)lam[FieldMap<T, 10>::at(j, f, L.fs)];
        v[0] -= kCs2 * (v[4] + v[5] + v[6]);
        for (int f = 0; f < 10; ++f) {
            if (dt == LLB_F64) static_cast<double*>(g)[f * N + i] = v[f];
            else static_cast<float*>(g)[f * N + i] = (float)v[f];
        }
    }
}

// Two components: canonical (rho1, rho2, j, P) <-> internal (rho1, d, j, A) with
// rho2 = 1 + d - rho1, P_aa = A_aa + cs^2 (1 + d); cotangents map by the transposes.
template <class T>
__global__ void k_cot2_canon_to_internal(const void* __restrict__ g, int dt, T* __restrict__ lam, Layout L) {
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        double v[11];
        for (int f = 0; f < 11; ++f)
            v[f] = dt == LLB_F64 ? static_cast<const double*>(g)[f * N + i] : (double)static_cast<const float*>(g)[f * N + i];
        const int x = (int)(i % L.nx);
        const size_t r = i / L.nx;
        const size_t j = L.at(x, (int)(r % L.ny), (int)(r / L.ny));
        lam[j] = (T)(v[0] - v[1]);
        lam[L.fs + j] = (T)(v[1] + kCs2 * (v[5] + v[6] + v[7]));
        for (int f = 2; f < 11; ++f) lam[f * L.fs + j] = (T)v[f];
    }
}

template <class T>
__global__ void k_cot2_internal_to_canon(const T* __restrict__ lam, void* __restrict__ g, int dt, Layout L) {
    const size_t N = (size_t)L.nx * L.ny * L.nz;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % L.nx);
        const size_t r = i / L.nx;
        const size_t j = L.at(x, (int)(r % L.ny), (int)(r / L.ny));
        double v[11];
        for (int f = 0; f < 11; ++f) v[f] = (double)lam[f * L.fs + j];
        const double tr = kCs2 * (v[5] + v[6] + v[7]);
        const double g1 = v[0] + v[1] - tr, g2 = v[1] - tr;
        v[0] = g1;
        v[1] = g2;
        for (int f = 0; f < 11; ++f) {
            if (dt == LLB_F64) static_cast<double*>(g)[f * N + i] = v[f];
            else static_cast<float*>(g)[f * N + i] = (float)v[f];
        }
    }
}

dim3 adj_grid(const llb_ctx& c) { return dim3((c.nx + kAdjThreads - 1) / kAdjThreads, c.ny, c.nz); }

// Three CTAs of four warps per SM: 168 registers, of which the pull, two nodes' state and
// the loads ahead take all (four CTAs: spills).
constexpr int kAdjCtas = 3;

template <class L, class T>
cudaError_t adj_step_t(const llb_ctx& c, const void* lam_new, const void* m, void* lam, double* rows, size_t* nrows) {
    if constexpr (std::is_same<T, float>::value) {
        using K = mom::PairTile<L, mom::kPairH>;
        auto kern = mom::k_moment_pair<L, float, mom::kPairH, kAdjCtas, Adjoint<L>>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, K::g_bytes);
        int per_sm = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, K::NT, K::g_bytes);
        if (e != cudaSuccess) return e;
        const int fit = std::max(per_sm, 1) * c.num_sms;
        const mom::Sched sc = mom::plan(c.nx, c.ny, c.nz, K::BX, K::BY, fit);
        *nrows = std::min(sc.nitems, fit);
        return launch_overlapped(kern, (int)*nrows, K::NT, K::g_bytes, c.stream, static_cast<const float*>(lam_new),
                                 static_cast<float*>(lam), c.lay, Adjoint<L>{static_cast<const float*>(m), (float)c.omega, rows},
                                 sc, 0, c.nz, 0, static_cast<int*>(nullptr));
    } else {
        k_adjoint_step<L, T><<<adj_grid(c), kAdjThreads, 0, c.stream>>>(static_cast<const T*>(lam_new),
                                                                         static_cast<const T*>(m), static_cast<T*>(lam),
                                                                         c.lay, (T)c.omega, rows);
        *nrows = (size_t)adj_grid(c).x * c.ny * c.nz;
        return cudaGetLastError();
    }
}

cudaError_t adj_step(const llb_ctx& c, const void* lam_new, const void* m, void* lam, double* rows, size_t* nrows) {
    if (c.Q == 19)
        return c.storage == LLB_F64 ? adj_step_t<D3Q19, double>(c, lam_new, m, lam, rows, nrows)
                                    : adj_step_t<D3Q19, float>(c, lam_new, m, lam, rows, nrows);
    return c.storage == LLB_F64 ? adj_step_t<D3Q27, double>(c, lam_new, m, lam, rows, nrows)
                                : adj_step_t<D3Q27, float>(c, lam_new, m, lam, rows, nrows);
}

// CTAs of the tiled first pass for this context (0 if it cannot run).
template <class L, class T>
int adj_tiled_ctas(const llb_ctx& c) {
    using C = AdjTile<L, T, kAdjBX, kAdjBY>;
    auto kern = k_adjoint_cg_tiled<L, T, kAdjBX, kAdjBY>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem_bytes) != cudaSuccess)
        return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::NT, C::smem_bytes) != cudaSuccess || per_sm < 1)
        return 0;
    const mom::Sched sc = mom::plan(c.nx, c.ny, c.nz, kAdjBX, kAdjBY, per_sm * c.num_sms);
    return std::min(sc.nitems, per_sm * c.num_sms);
}

// One two-component adjoint step; *nrows: rows of dL/domega partial sums written.
template <class L, class T>
cudaError_t adj_cg_step_t(const llb_ctx& c, const void* lam_new, const void* m, void* lam, void* lam_g,
                          double* rows, size_t* nrows) {
    CGAdjPar<T> p;
    p.omega = (T)c.omega;
    p.beta = (T)c.params.beta;
    p.A_s = (T)c.params.A_s;
    p.eps2 = (T)(c.params.grad_eps * c.params.grad_eps);
    const int grid = (c.params.debug_flags & 2) ? 0 : adj_tiled_ctas<L, T>(c);
    if (grid > 0) {
        using C = AdjTile<L, T, kAdjBX, kAdjBY>;
        const mom::Sched sc = mom::plan(c.nx, c.ny, c.nz, kAdjBX, kAdjBY, grid);
        k_adjoint_cg_tiled<L, T, kAdjBX, kAdjBY><<<grid, C::NT, C::smem_bytes, c.stream>>>(
            static_cast<const T*>(lam_new), static_cast<const T*>(m), static_cast<T*>(lam), static_cast<T*>(lam_g),
            c.lay, p, sc, rows);
        *nrows = (size_t)grid;
    } else {  // reference form: one thread per node, neighbour fields loaded directly
        k_adjoint_cg_local<L, T><<<adj_grid(c), kAdjThreads, 0, c.stream>>>(
            static_cast<const T*>(lam_new), static_cast<const T*>(m), static_cast<T*>(lam), static_cast<T*>(lam_g),
            c.lay, p, rows);
        *nrows = (size_t)adj_grid(c).x * c.ny * c.nz;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const dim3 phi_grid((c.nx + kPhiX - 1) / kPhiX, (c.ny + kPhiY - 1) / kPhiY, (c.nz + kPhiPlanes - 1) / kPhiPlanes);
    k_adjoint_cg_phi<L, T><<<phi_grid, dim3(kPhiX, kPhiY), 0, c.stream>>>(static_cast<const T*>(m),
                                                                      static_cast<const T*>(lam_g),
                                                                      static_cast<T*>(lam), c.lay);
    return cudaGetLastError();
}

cudaError_t adj_cg_step(const llb_ctx& c, const void* lam_new, const void* m, void* lam, void* lam_g, double* rows,
                        size_t* nrows) {
    if (c.Q == 19)
        return c.storage == LLB_F64 ? adj_cg_step_t<D3Q19, double>(c, lam_new, m, lam, lam_g, rows, nrows)
                                    : adj_cg_step_t<D3Q19, float>(c, lam_new, m, lam, lam_g, rows, nrows);
    return c.storage == LLB_F64 ? adj_cg_step_t<D3Q27, double>(c, lam_new, m, lam, lam_g, rows, nrows)
                                : adj_cg_step_t<D3Q27, float>(c, lam_new, m, lam, lam_g, rows, nrows);
}

int grid_n(const llb_ctx& c) {
    const size_t want = (c.N + 255) / 256;
    const size_t cap = (size_t)(c.num_sms > 0 ? c.num_sms : 148) * 8;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// One forward step (same kernels as llb_step) from `in` to `out`.
cudaError_t fwd(const llb_ctx& c, const void* in, void* out) {
    return c.ncomp == 2                   ? launch_cg_tiled(c, in, out)
           : c.kernel == LLB_KERNEL_TMA   ? launch_moment_tma(c, c.cur, out)
           : c.kernel == LLB_KERNEL_TILED ? launch_moment_tiled(c, c.cur, in, out, false)
                                          : launch_moment_direct(c, in, out);
}

// Whether fwd takes any pair of state buffers: the TMA-staged kernel and the L2
// prefetch of tiled variant 1 hold tensor maps of the context's own two buffers.
bool any_buffer(const llb_ctx& c) {
    return c.ncomp == 2 || c.kernel == LLB_KERNEL_DIRECT || (c.kernel == LLB_KERNEL_TILED && c.variant != 1);
}

// Advance the context by one step, flipping cur.
cudaError_t fwd_one(llb_ctx* c) {
    const cudaError_t e = fwd(*c, c->buf[c->cur], c->buf[1 - c->cur]);
    if (e == cudaSuccess) c->cur = 1 - c->cur;
    return e;
}

}  // namespace

LLB_CHK_TU(adjoint)

}  // namespace llb

namespace llb {
namespace {

// Device memory of one adjoint call, in the order it is laid out (256-byte pieces).
// Where the step takes any pair of buffers the starting state is the context's own and
// stays in place, so segment 0 needs no checkpoint and a segment no copy of its first
// state; the others hold a copy of both.
struct AdjWork {
    int K, nseg, nck, nslot;
    size_t sb, nrows, ck, seg, lamA, lamB, lamG, rows, acc, bytes;

    AdjWork(const llb_ctx& c, int nsteps, int every) {
        K = every > 0 ? every : (int)std::fmax(1.0, std::round(std::sqrt((double)nsteps)));
        nseg = nsteps > 0 ? (nsteps + K - 1) / K : 0;
        const bool direct = any_buffer(c);
        nck = direct ? std::max(nseg - 1, 0) : nseg;
        nslot = std::min(K, nsteps) - (direct ? 1 : 0);
        // rows of dL/domega partial sums: one per block of the one-thread-per-node kernels,
        // or one per CTA of the tiled first pass (at most 32 per SM)
        nrows = std::max((size_t)adj_grid(c).x * c.ny * c.nz, (size_t)32 * (c.num_sms > 0 ? c.num_sms : 1));
        bytes = 0;
        auto piece = [&](size_t n) {
            const size_t at = bytes;
            bytes += (n + 255) / 256 * 256;
            return at;
        };
        sb = (c.state_bytes + 255) / 256 * 256;
        ck = piece(sb * (size_t)nck);
        seg = piece(sb * (size_t)std::max(nslot, 0));
        lamA = piece(sb);
        lamB = piece(sb);
        lamG = c.ncomp == 2 ? piece(sb) : lamA;  // cotangent of G (3 fields), two components only
        rows = piece(nrows * sizeof(double));
        acc = piece(sizeof(double));
    }
};

bool adjoint_takes(const llb_ctx& c, int nsteps) {
    if (c.in_batch || c.scheme != LLB_SCHEME_MOMENT || (c.storage != LLB_F32 && c.storage != LLB_F64) || nsteps < 0)
        return false;
    // two components: differentiable only without the near-contact switch and with the smooth normal
    return c.ncomp != 2 || (c.params.A_h == 0.0 && c.params.grad_eps > 0.0);
}

}  // namespace
}  // namespace llb

extern "C" int llb_adjoint(llb_ctx* c, int nsteps, int every, const void* dev_gfinal, void* dev_ginit, int dtype,
                           double* dtau) {
    return llb_adjoint_in(c, nsteps, every, dev_gfinal, dev_ginit, dtype, dtau, nullptr, 0);
}

extern "C" int llb_adjoint_bytes(const llb_ctx* c, int nsteps, int every, size_t* out) {
    if (!c || !out || !llb::adjoint_takes(*c, nsteps)) return LLB_EINVAL;
    *out = llb::AdjWork(*c, nsteps, every).bytes;
    return LLB_OK;
}

extern "C" int llb_adjoint_in(llb_ctx* c, int nsteps, int every, const void* dev_gfinal, void* dev_ginit, int dtype,
                              double* dtau, void* work, size_t work_bytes) {
    using namespace llb;
    if (!c) return LLB_EINVAL;
    if (c->sticky != LLB_OK) return LLB_ESTATE;
    if (!adjoint_takes(*c, nsteps) || !dev_gfinal || !dev_ginit || (dtype != LLB_F64 && dtype != LLB_F32))
        return LLB_EINVAL;
    const bool two = c->ncomp == 2;
    const AdjWork w(*c, nsteps, every);
    const int K = w.K, nseg = w.nseg;
    const size_t sb = w.sb;
    if (work && (work_bytes < w.bytes || reinterpret_cast<uintptr_t>(work) % 256 != 0)) return LLB_EINVAL;
    void* own = nullptr;
    if (!work && cudaMalloc(&own, w.bytes) != cudaSuccess) {
        cudaGetLastError();
        return LLB_ENOMEM;
    }
    auto release = [&]() {
        cudaStreamSynchronize(c->stream);
        if (own) cudaFree(own);
        cudaGetLastError();
    };
    char* const base = static_cast<char*>(work ? work : own);
    char *const ck = base + w.ck, *const seg = base + w.seg;
    void *const lamA = base + w.lamA, *const lamB = base + w.lamB, *const lamG = base + w.lamG;
    double *const rows = reinterpret_cast<double*>(base + w.rows), *const acc = reinterpret_cast<double*>(base + w.acc);
    const size_t nrows = w.nrows;
    const int cur0 = c->cur;
    const long long t0 = c->t;
    cudaError_t e = cudaMemsetAsync(acc, 0, sizeof(double), c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(rows, 0, nrows * sizeof(double), c->stream);
    // State s of the trajectory where the step takes any pair of buffers: the context's
    // own, a checkpoint (every K steps) or a slot of the segment at hand.
    const bool direct = any_buffer(*c);
    auto state = [&](int s) -> char* {
        if (!direct) return seg + (size_t)(s % K) * sb;
        if (s == 0) return static_cast<char*>(c->buf[cur0]);
        return s % K == 0 ? ck + (size_t)(s / K - 1) * sb : seg + (size_t)(s % K - 1) * sb;
    };
    // forward to the last state the sweep reads, nsteps - 1: the slots then hold the last segment
    for (int s = 0; s + 1 < nsteps && e == cudaSuccess && direct; ++s) e = fwd(*c, state(s), state(s + 1));
    // other steps: in the context's buffers, up to the last checkpoint
    for (int s = 0; s < nsteps && e == cudaSuccess && !direct; ++s) {
        if (s % K == 0)
            e = cudaMemcpyAsync(ck + (size_t)(s / K) * sb, c->buf[c->cur], c->state_bytes, cudaMemcpyDeviceToDevice,
                                c->stream);
        if (s == (nseg - 1) * K) break;
        if (e == cudaSuccess) e = fwd_one(c);
    }
    // cotangent of the final state
    if (e == cudaSuccess) {
        if (two && c->storage == LLB_F64)
            k_cot2_canon_to_internal<double><<<grid_n(*c), 256, 0, c->stream>>>(dev_gfinal, dtype, static_cast<double*>(lamA), c->lay);
        else if (two)
            k_cot2_canon_to_internal<float><<<grid_n(*c), 256, 0, c->stream>>>(dev_gfinal, dtype, static_cast<float*>(lamA), c->lay);
        else if (c->storage == LLB_F64)
            k_cot_canon_to_shifted<double><<<grid_n(*c), 256, 0, c->stream>>>(dev_gfinal, dtype, static_cast<double*>(lamA), c->lay);
        else
            k_cot_canon_to_shifted<float><<<grid_n(*c), 256, 0, c->stream>>>(dev_gfinal, dtype, static_cast<float*>(lamA), c->lay);
        e = cudaGetLastError();
    }
    void* lam_in = lamA;
    void* lam_out = lamB;
    // every block adds its dL/domega of each step to its own row; the rows are summed once, at the end
    size_t used = (size_t)adj_grid(*c).x * c->ny * c->nz;
    for (int k = nseg - 1; k >= 0 && e == cudaSuccess; --k) {
        const int s0 = k * K, s1 = s0 + K < nsteps ? s0 + K : nsteps;
        // recompute the states s0 .. s1-1 of this segment from its checkpoint
        if (direct) {
            for (int s = s0; s + 1 < s1 && e == cudaSuccess && k < nseg - 1; ++s) e = fwd(*c, state(s), state(s + 1));
        } else {
            e = cudaMemcpyAsync(c->buf[c->cur], ck + (size_t)k * sb, c->state_bytes, cudaMemcpyDeviceToDevice, c->stream);
            for (int s = s0; s < s1 && e == cudaSuccess; ++s) {
                e = cudaMemcpyAsync(state(s), c->buf[c->cur], c->state_bytes, cudaMemcpyDeviceToDevice, c->stream);
                if (e == cudaSuccess && s + 1 < s1) e = fwd_one(c);
            }
        }
        for (int s = s1 - 1; s >= s0 && e == cudaSuccess; --s) {
            e = two ? adj_cg_step(*c, lam_in, state(s), lam_out, lamG, rows, &used)
                    : adj_step(*c, lam_in, state(s), lam_out, rows, &used);
            void* tmp = lam_in;
            lam_in = lam_out;
            lam_out = tmp;
        }
    }
    if (e == cudaSuccess) {
        k_sum_rows<<<1, 256, 0, c->stream>>>(rows, used, acc);
        e = cudaGetLastError();
    }
    // cotangent of the initial state, in canonical form
    if (e == cudaSuccess) {
        if (two && c->storage == LLB_F64)
            k_cot2_internal_to_canon<double><<<grid_n(*c), 256, 0, c->stream>>>(static_cast<const double*>(lam_in), dev_ginit, dtype, c->lay);
        else if (two)
            k_cot2_internal_to_canon<float><<<grid_n(*c), 256, 0, c->stream>>>(static_cast<const float*>(lam_in), dev_ginit, dtype, c->lay);
        else if (c->storage == LLB_F64)
            k_cot_shifted_to_canon<double><<<grid_n(*c), 256, 0, c->stream>>>(static_cast<const double*>(lam_in), dev_ginit, dtype, c->lay);
        else
            k_cot_shifted_to_canon<float><<<grid_n(*c), 256, 0, c->stream>>>(static_cast<const float*>(lam_in), dev_ginit, dtype, c->lay);
        e = cudaGetLastError();
    }
    double domega = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&domega, acc, sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    // the error word of the forward steps: this call synchronises, so it reports a wait that gave up
    int gave_up = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&gave_up, c->err_dev, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
    // restore the initial state
    if (e == cudaSuccess && nseg > 0 && !direct)
        e = cudaMemcpyAsync(c->buf[cur0], ck, c->state_bytes, cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    c->cur = cur0;
    c->t = t0;
    release();
    if (e != cudaSuccess) {
        c->sticky = LLB_ECUDA;
        c->msg = std::string("adjoint: ") + cudaGetErrorString(e);
        return LLB_ECUDA;
    }
    if (gave_up) {
        c->sticky = LLB_ETIMEOUT;
        c->msg = "adjoint: a device wait gave up (a TMA load or a plane barrier did not complete)";
        return LLB_ETIMEOUT;
    }
    // omega = 1 / tau
    if (dtau) *dtau = -domega / (c->tau * c->tau);
    return LLB_OK;
}
