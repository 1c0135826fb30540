// One-component moment-only step, FP32 arithmetic, two nodes per thread
// (pair_march.cuh).
//
// The march of moment_tiled.cuh with the work of a thread doubled.  The one-node
// form executed 334 thread-instructions per node on D3Q19 at half the issue rate,
// with 4.4 of 8 warps colliding a halo node per plane; the pair executes
// 219 and a CTA's halo is one warp.
//
// A CTA is H tile warps and a halo warp for the rows above and below.  A warp
// holds 32 columns, the inner 30 its outputs: the outer two are collided for
// their populations only.  (32 outputs per warp and the side columns loaded by
// themselves was slower: such a load touches one sector of a line per lane, and
// the load pipe, 60 to 70 % busy, spends as much on it as on the tile.)  The rows above
// and below are doubled in the exchange (one copy for every other plane), so that
// the halo warp publishes plane s + 1 while the tile warps still pull plane s;
// doubling all of it costs the L1 space that the loads in flight need (256^3: 404
// against 350 us of an earlier form).
#pragma once

#include <algorithm>

#include "moment_common.cuh"
#include "overlap.cuh"
#include "pair_march.cuh"

namespace llb {
namespace mom {

// Constants of the scaled collision (host side, FP64, rounded once).  The
// stored element of field f is the moment times narrow_scale(f) in a 16-bit
// state; the factors below undo it.
struct CollK {
    float d1;          // density deviation of a stored d
    float ka, kc, ko;  // 4.5 w (1 - omega), 9 w (1 - omega), 4.5 w omega
    float wd, wj, wj2; // w, 3 w and what rounding it left
};

template <class L, class S>
CollK coll_constants(double omega) {
    const double w = pk::Shells<L>::w;
    const bool n = IsNarrow<S>::value;
    const double sd = n ? narrow_scale(0) : 1.0, sj = n ? narrow_scale(1) : 1.0, sa = n ? narrow_scale(4) : 1.0;
    CollK k;
    k.d1 = (float)(1.0 / sd);
    k.ka = (float)(4.5 * w * (1.0 - omega) / sa);
    k.kc = (float)(9.0 * w * (1.0 - omega) / sa);
    k.ko = (float)(4.5 * w * omega / (sj * sj));
    k.wd = (float)(w / sd);
    k.wj = (float)(3.0 * w / sj);
    k.wj2 = (float)(3.0 * w / sj - (double)k.wj);
    return k;
}

template <class V>
__device__ __forceinline__ pk::Col<V> collide_scaled(const V* v, const CollK& k) {
    using namespace pk;
    const V r = mul(k.ko, rcp1p(k.d1, v[0]));
    const V ox = mul(r, v[1]), oy = mul(r, v[2]), oz = mul(r, v[3]);
    const V tx = add(ox, ox), ty = add(oy, oy);
    Col<V> c;
    c.xx = fma(ox, v[1], mul(k.ka, v[4]));
    c.yy = fma(oy, v[2], mul(k.ka, v[5]));
    c.zz = fma(oz, v[3], mul(k.ka, v[6]));
    c.xy = fma(tx, v[2], mul(k.kc, v[7]));
    c.xz = fma(tx, v[3], mul(k.kc, v[8]));
    c.yz = fma(ty, v[3], mul(k.kc, v[9]));
    c.jx = col_j(k.wj, k.wj2, v[1]);
    c.jy = col_j(k.wj, k.wj2, v[2]);
    c.jz = col_j(k.wj, k.wj2, v[3]);
    c.s = col_s(c.xx, c.yy, c.zz, mul(k.wd, v[0]));
    return c;
}

template <class L, int H_>
struct PairTile {
    static constexpr int W = 32, BX = W - 2, H = H_, BY = 2 * H_;
    static constexpr int NT = W * (H + 1);   // H tile warps and the halo warp
    // pair slots of one direction: rows 0 .. H-1, two copies of the row above and two of the row below
    static constexpr int HN = W * (H + 4);
    static constexpr bool kC = pk::Shells<L>::corners;
    static constexpr int N4 = kC ? 8 : 4, N2 = kC ? 0 : 4;  // directions with (c0, c1), with c0 only
    static constexpr int g_bytes = HN * (16 * N4 + 8 * (N2 + 1));
};

// Pair of the elements of two nodes.
template <class S>
__device__ __forceinline__ float2 widen(S lo, S hi) {
    if constexpr (std::is_same<S, __half>::value) return make_float2(__half2float(lo), __half2float(hi));
    else if constexpr (std::is_same<S, __nv_bfloat16>::value)
        return make_float2(__bfloat162float(lo), __bfloat162float(hi));
    else return make_float2(lo, hi);
}

// Store field f of a pair (in the stored scale already) at the two nodes.
template <class S>
__device__ __forceinline__ void narrow(float2 v, S& lo, S& hi) {
    if constexpr (std::is_same<S, __half>::value) {
        const __half2 h = __floats2half2_rn(v.x, v.y);
        lo = __low2half(h);
        hi = __high2half(h);
    } else if constexpr (std::is_same<S, __nv_bfloat16>::value) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
        lo = __low2bfloat16(h);
        hi = __high2bfloat16(h);
    } else {
        lo = v.x;
        hi = v.y;
    }
}

// Periodic ghost copies of node (x, y) whose ten stored elements are v (y_only:
// without the copy in x alone): the copies that exist are the set bits of a
// mask, so a node at one face runs one iteration.
template <class S>
__device__ __forceinline__ void store_ghosts(S* out, const Layout& lay, int x, int y, int z, const S* v, bool y_only) {
    const unsigned xm = (x < kGhostX ? 1u : 0u) | (x >= lay.nx - kGhostX ? 2u : 0u);
    const unsigned ym = (y < lay.yo ? 1u : 0u) | (y >= lay.ny - lay.yo ? 2u : 0u);
    // copy k = 3 yk + xk: shift by 0, +n, -n in each direction
    unsigned todo = (xm << 1) | (ym & 1u ? ((xm << 1) | 1u) << 3 : 0u) | (ym & 2u ? ((xm << 1) | 1u) << 6 : 0u);
    if (y_only) todo &= ~7u;
    while (todo) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1;
        const int xk = k % 3, yk = k / 3;
        const int gx = x + (xk == 1 ? lay.nx : xk == 2 ? -lay.nx : 0);
        const int gy = y + (yk == 1 ? lay.ny : yk == 2 ? -lay.ny : 0);
        const size_t i = lay.at(gx, gy, z);
        if (!LLB_IN(i, lay.fs, kChkGhost)) continue;
#pragma unroll
        for (int f = 0; f < 10; ++f) out[FieldMap<S, 10>::at(i, f, lay.fs)] = v[f];
    }
}

// What the march computes: the step itself (Step), or the adjoint of a step, whose
// streaming is the same with the directions reversed (Adjoint, adjoint.cu).
template <class S>
struct Step {
    static constexpr bool kAdjoint = false;
    CollK k;
    struct Sum {};
    __device__ __forceinline__ pk::Col<float2> column(const float2* v) const { return collide_scaled(v, k); }
};

template <class L, class S, int H, int MINB, class Op>
__global__ void __launch_bounds__(32 * (H + 1), MINB)
    k_moment_pair(const S* in, S* out, Layout lay, Op op, Sched sc, int zlo, int nzr, int ghosts, int* queue) {
    using namespace pk;
    using K = PairTile<L, H>;
    using SH = Shells<L>;
    constexpr bool kC = K::kC;
    constexpr int W = K::W, BX = K::BX, HN = K::HN, BY = K::BY;
    constexpr bool IL = FieldMap<S, 10>::kInterleaved;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* const G4 = reinterpret_cast<float4*>(smem_raw);             // (c0 lo, c0 hi, c1 lo, c1 hi) per direction
    float2* const GZ = reinterpret_cast<float2*>(G4 + K::N4 * HN);      // zz
    float2* const G2 = GZ + HN;                                         // c0 of the diagonals (D3Q19)
    float* const F4 = reinterpret_cast<float*>(G4);
    float* const FZ = reinterpret_cast<float*>(GZ);
    float* const F2 = reinterpret_cast<float*>(G2);
    const int nx = lay.nx, ny = lay.ny, nz = lay.nz;
    const size_t fs = IL ? 32 : lay.fs;                            // elements between the fields of a node
    const size_t plane = (size_t)lay.px * lay.py * (IL ? 10 : 1);  // elements between planes (a field's, or all)
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto elem = [&](int x, int y) { return FieldMap<S, 10>::at(lay.at(pmod(x, nx), pmod(y, ny), 0), 0, lay.fs); };
    auto load = [&](S* v, size_t e) {
        if (LLB_IN(e + 9 * fs, 10 * lay.fs, kChkLoad)) {
#pragma unroll
            for (int f = 0; f < 10; ++f) v[f] = load_dep(in + e + f * fs);
        }
    };
    const float2 zero = make_float2(0.0f, 0.0f);
    int par = 0;  // parity of the plane: which copy of the halo slots it uses

    // Items: the first by block index, the others from a queue (queue[0]: items taken
    // beyond the first round, queue[1]: CTAs done), asked for when an item begins.  The
    // last CTA to leave resets it for the next launch.  The adjoint takes them round-robin,
    // so that its sum over the nodes has one order.
    __shared__ int s_next;
    typename Op::Sum total;
    dep_wait();
    for (int it = blockIdx.x; it < sc.nitems;) {
        if (threadIdx.x == 0)
            s_next = Op::kAdjoint ? it + (int)gridDim.x : (int)gridDim.x + (sc.nitems > (int)gridDim.x ? atomicAdd(queue, 1) : sc.nitems);
        int x0, y0, za, zb;  // outputs za .. zb-1 of the tile at (x0, y0)
        sc.item(it, BX, BY, nzr, x0, y0, za, zb);
        za += zlo;
        zb += zlo;
        int zn = pmod(za - 1, nz);  // source plane of the next load
        size_t zo = (size_t)zn * plane;
        auto advance = [&]() {
            if (++zn == nz) {
                zn = 0;
                zo = 0;
            } else {
                zo += plane;
            }
        };

        const int ox = x0 - 1 + lane;  // column of this lane

        if (w == H) {
            // ---- halo warp: the rows above and below the tile, the row below
            // mirrored in y, so that c_y = +1 enters the tile from both
            const size_t e0 = elem(ox, y0 - 1), e1 = elem(ox, y0 + BY);
            S a0[10], a1[10];
            load(a0, e0 + zo);
            load(a1, e1 + zo);
#pragma unroll 1
            for (int s = za - 1;; ++s) {
                const bool more = s < zb;
                if (more) advance();
                float2 v[10];
#pragma unroll
                for (int f = 0; f < 10; ++f) v[f] = widen(a0[f], a1[f]);
                Col<float2> c = op.column(v);
                if (more) {
                    load(a0, e0 + zo);
                    load(a1, e1 + zo);
                }
                c.jy.y = -c.jy.y;
                c.xy.y = -c.xy.y;
                c.yz.y = -c.yz.y;
                const int gt = (H + par) * W + lane, gb = (H + 2 + par) * W + lane;
                emit_plane(c, [](int, int cy) { return cy == 1; }, [&](auto d, float2 c0, float2 c1) {
                    using D = decltype(d);
                    constexpr int kt = plane_dir(D::cx, 1), kb = plane_dir(D::cx, -1);
                    if constexpr (kC || D::cx == 0) {
                        F4[4 * (kt * HN + gt)] = c0.x;
                        F4[4 * (kt * HN + gt) + 2] = c1.x;
                        F4[4 * (kb * HN + gb) + 1] = c0.y;
                        F4[4 * (kb * HN + gb) + 3] = c1.y;
                    } else {
                        F2[2 * ((kt - 4) * HN + gt)] = c0.x;
                        F2[2 * ((kb - 4) * HN + gb) + 1] = c0.y;
                    }
                });
                FZ[2 * gt] = c.zz.x;
                FZ[2 * gb + 1] = c.zz.y;
                par ^= 1;
                bar_sync<1, K::NT>();  // the exchange of plane s is complete
                if (!more) break;
            }
            __syncthreads();
            it = s_next;
            __syncthreads();
            continue;
        }

        // ---- tile warp: pair row w, column lane
        const int n1 = w * W + lane;
        const int oy = y0 + w;
        const bool ok_x = lane >= 1 && lane <= BX && ox < nx;
        const bool ok_lo = ok_x && oy < ny, ok_hi = ok_x && oy + H < ny;
        const size_t e_lo = elem(ox, oy), e_hi = elem(ox, oy + H);
        // Periodic ghost copies.  A box of at least 16 x 2 nodes gives a node at most
        // one copy in x (8 columns beyond the opposite face) and one in y (the whole
        // row), at distances that are the same in every plane and, in x, every row;
        // smaller boxes take the general store_ghosts.
        const bool gsmall = nx < 2 * kGhostX || ny < 2;
        // (+-nx in a field-major state, where 64 bits cost spilled registers on D3Q27)
        const auto gdx = [&] {
            if constexpr (IL) return ok_x ? ghost_shift_x<S, 10>(lay, ox) : std::ptrdiff_t(0);
            else return ox < kGhostX ? nx : ox >= nx - kGhostX ? -nx : 0;
        }();
        const bool gy = oy < lay.yo || oy >= ny - lay.yo || oy + H >= ny - lay.yo;  // a row with a copy, warp-uniform
        S lo[10], hi[10];
        load(lo, e_lo + zo);
        load(hi, e_hi + zo);

        // rolling sums: of the plane ahead of the source plane (its c_z = +1
        // pulls), and of the source plane (those and its c_z = 0 pulls; the
        // former's g, jx, jy also carry the c_z moments)
        PlaneSum<float2> P{zero, zero, zero, zero, zero, zero}, A{zero, zero, zero, zero, zero, zero};
        float2 zg = zero, zx = zero, zy = zero;

#pragma unroll 1
        for (int s = za - 1;; ++s) {
            const bool more = s < zb;
            if (more) advance();
            float2 own_s, own_z, own_zz;
            {
                float2 v[10];
#pragma unroll
                for (int f = 0; f < 10; ++f) v[f] = widen(lo[f], hi[f]);
                const Col<float2> c = op.column(v);
                if (more) {
                    load(lo, e_lo + zo);
                    load(hi, e_hi + zo);
                }
                own_s = c.s;
                own_z = c.jz;
                own_zz = c.zz;
                if (LLB_IN(n1, HN, kChkPublish)) {
                    const int up = (H + par) * W + lane, dn = (H + 2 + par) * W + lane;
                    emit_plane(c, [](int, int) { return true; }, [&](auto d, float2 c0, float2 c1) {
                        using D = decltype(d);
                        constexpr int kk = plane_dir(D::cx, D::cy);
                        if constexpr (kk < K::N4) {
                            G4[kk * HN + n1] = make_float4(c0.x, c0.y, c1.x, c1.y);
                            if (D::cy > 0 && w == H - 1) {
                                F4[4 * (kk * HN + up) + 1] = c0.x;
                                F4[4 * (kk * HN + up) + 3] = c1.x;
                            }
                            if (D::cy < 0 && w == 0) {
                                F4[4 * (kk * HN + dn)] = c0.y;
                                F4[4 * (kk * HN + dn) + 2] = c1.y;
                            }
                        } else {
                            G2[(kk - 4) * HN + n1] = c0;
                            if (D::cy > 0 && w == H - 1) F2[2 * ((kk - 4) * HN + up) + 1] = c0.x;
                            if (D::cy < 0 && w == 0) F2[2 * ((kk - 4) * HN + dn)] = c0.y;
                        }
                    });
                    GZ[n1] = c.zz;
                    if (w == H - 1) FZ[2 * up + 1] = c.zz.x;
                    if (w == 0) FZ[2 * dn] = c.zz.y;
                }
            }
            // the state at the output nodes, for the adjoint
            S ml[Op::kAdjoint ? 10 : 1], mh[Op::kAdjoint ? 10 : 1];
            if constexpr (Op::kAdjoint) {
                if (s > za) {
                    const size_t zw = (size_t)(s - 1) * plane;
                    op.load(ml, e_lo + zw, fs, lay.fs);
                    op.load(mh, e_hi + zw, fs, lay.fs);
                }
            }
            bar_sync<1, K::NT>();  // the exchange of plane s is complete
            // slots of the neighbours: rows y - 1, y + 1 and columns x - 1, x + 1
            const int up = (w == 0 ? H + par : w - 1) * W, dn = (w == H - 1 ? H + 2 + par : w + 1) * W, mid = w * W;
            const int lf = max(lane - 1, 0), rt = min(lane + 1, W - 1);
            par ^= 1;
            auto at = [&](int row, int col) { return LLB_IN(row + col, HN, kChkGather) ? row + col : 0; };
            const int nl = at(mid, lf), nr = at(mid, rt), nu = at(up, lane), nd = at(dn, lane);
            const int nul = at(up, lf), nur = at(up, rt), ndl = at(dn, lf), ndr = at(dn, rt);
            // shell factors; those of D3Q27's c_z = 0 plane are 4 times the other planes' and applied last
            constexpr float s0 = kC ? 4.0f : 1.0f, o0 = SH::own0 / s0, a0 = SH::axis0 / s0, o1 = SH::own1, a1 = SH::axis1;
            struct Nb {
                float2 c0, c1, t;
            };
            auto nb = [&](int kk, int n) {
                const float4 c = G4[kk * HN + n];
                const float2 c0 = make_float2(c.x, c.y);
                return Nb{c0, make_float2(c.z, c.w), add(c0, GZ[n])};
            };
            const Nb l = nb(0, nl), r1 = nb(1, nr), u = nb(2, nu), d = nb(3, nd);
            const float2 own_t = add(own_s, own_zz);
            PlaneSum<float2> q0, qt, qc;
            if constexpr (kC) {
                const Nb pp = nb(4, nul), mm = nb(5, ndr), pm = nb(6, ndl), mp = nb(7, nur);
                qt = plane_sum<true>(o1, a1, 1.0f, own_t, l.t, r1.t, u.t, d.t, pp.t, mm.t, pm.t, mp.t);
                qc = plane_sum<true>(o1, a1, 1.0f, own_z, l.c1, r1.c1, u.c1, d.c1, pp.c1, mm.c1, pm.c1, mp.c1);
                q0 = plane_sum<true>(o0, a0, 1.0f, own_s, l.c0, r1.c0, u.c0, d.c0, pp.c0, mm.c0, pm.c0, mp.c0);
            } else {
                qt = plane_sum<false>(o1, a1, 1.0f, own_t, l.t, r1.t, u.t, d.t, zero, zero, zero, zero);
                qc = plane_sum<false>(o1, a1, 1.0f, own_z, l.c1, r1.c1, u.c1, d.c1, zero, zero, zero, zero);
                q0 = plane_sum<true>(o0, a0, 1.0f, own_s, l.c0, r1.c0, u.c0, d.c0, G2[nul], G2[HN + ndr], G2[2 * HN + ndl],
                                     G2[3 * HN + nur]);
            }
            float2 r[10];  // plane s - 1 is complete with the c_z = -1 pulls, qt - qc
            const float2 g = sub(qt.g, qc.g), jx = sub(qt.jx, qc.jx), jy = sub(qt.jy, qc.jy);
            r[0] = add(A.g, g);
            r[1] = add(A.jx, jx);
            r[2] = add(A.jy, jy);
            r[3] = sub(zg, g);
            r[4] = add(A.xx, sub(qt.xx, qc.xx));
            r[5] = add(A.yy, sub(qt.yy, qc.yy));
            r[6] = add(zg, g);
            r[7] = kC ? add(A.xy, sub(qt.xy, qc.xy)) : A.xy;
            r[8] = sub(zx, jx);
            r[9] = sub(zy, jy);
            if constexpr (Op::kAdjoint) {
                if (s > za && (ok_lo || ok_hi)) op.finish(r, ml, mh, ok_lo, ok_hi, total);
            } else {
                const float third = (float)kCs2;
#pragma unroll
                for (int f = 4; f < 7; ++f) r[f] = fma(-third, r[0], r[f]);
            }
            if (s > za && (ok_lo || ok_hi)) {
                S a[10], b[10];
#pragma unroll
                for (int f = 0; f < 10; ++f)
                    narrow(IsNarrow<S>::value ? mul(narrow_scale(f), r[f]) : r[f], a[f], b[f]);
                const size_t zw = (size_t)(s - 1) * plane;
                auto store = [&](size_t e, const S* v) {
                    if (!LLB_IN(e + 9 * fs, 10 * lay.fs, kChkStore)) return;
#pragma unroll
                    for (int f = 0; f < 10; ++f) out[e + f * fs] = v[f];
                };
                if (ok_lo) store(e_lo + zw, a);
                if (ok_hi) store(e_hi + zw, b);
                if (ghosts && gdx && !gsmall) {
                    if (ok_lo) store(e_lo + zw + (size_t)gdx, a);
                    if (ok_hi) store(e_hi + zw + (size_t)gdx, b);
                }
                if (ghosts && (gy || gsmall)) {
                    if (ok_lo) store_ghosts(out, lay, ox, oy, s - 1, a, !gsmall);
                    if (ok_hi) store_ghosts(out, lay, ox, oy + H, s - 1, b, !gsmall);
                }
            }
            zg = P.g;
            zx = P.jx;
            zy = P.jy;
            A.g = fma(s0, q0.g, P.g);
            A.jx = fma(s0, q0.jx, P.jx);
            A.jy = fma(s0, q0.jy, P.jy);
            A.xx = fma(s0, q0.xx, P.xx);
            A.yy = fma(s0, q0.yy, P.yy);
            A.xy = kC ? fma(s0, q0.xy, P.xy) : q0.xy;
            P.g = add(qt.g, qc.g);
            P.jx = add(qt.jx, qc.jx);
            P.jy = add(qt.jy, qc.jy);
            P.xx = add(qt.xx, qc.xx);
            P.yy = add(qt.yy, qc.yy);
            if constexpr (kC) P.xy = add(qt.xy, qc.xy);
            bar_sync<2, 32 * H>();  // and read
            if (!more) break;
        }
        __syncthreads();
        it = s_next;
        __syncthreads();
    }
    dep_launch();
    if constexpr (Op::kAdjoint) op.end(total);
    if (!Op::kAdjoint && threadIdx.x == 0 && atomicAdd(queue + 1, 1) == (int)gridDim.x - 1) {
        queue[0] = 0;
        queue[1] = 0;
    }
}

// Tiles of 30 x 6, four CTAs of four warps per SM (128 registers at most, no spills).
// Measured without / with ghost copies, us per step, launched without overlap: 256^3 D3Q19 267 / 277, D3Q27 290 /
// 303; 192^3 D3Q19 FP16 113 / 127; 131 x 97 x 75 D3Q27 24.6 / 28.7 (one node per
// thread, with them in every step: 305, 342, 137, 35).  Two CTAs of eight warps (30 x 14):
// 263 / 283, 300 / 324, 111 / 141, 26.8 / 32.8.  Overlapped and without: 267, 288, 109, 22.2.
constexpr int kPairH = 3, kPairCtas = 4;

// Chunk length of a box whose items go through the queue.  Without ghost copies all
// items cost the same and should fill whole rounds; with them the items at the faces
// take longer, so they are made short enough that the queue evens them out.
inline Sched pair_plan(const llb_ctx& c, int nzr, int BX, int BY, int grid, bool ghosts) {
    Sched s = plan(c.nx, c.ny, nzr, BX, BY, grid);
    if (!ghosts || s.nitems <= grid) return s;
    double best = -1.0;
    for (int nch = 1; nch <= nzr; ++nch) {
        const int zc = (nzr + nch - 1) / nch, chunks = (nzr + zc - 1) / zc;
        const long long items = (long long)s.ntiles * chunks;
        if (items > (1LL << 30)) break;
        const double cost = ((double)items / grid + 0.7) * (zc + 2);
        if (best < 0.0 || cost < best) {
            best = cost;
            s.zc = zc;
            s.nitems = (int)items;
        }
    }
    return s;
}

template <class L, class S>
int pair_ctas(const llb_ctx& c) {
    using K = PairTile<L, kPairH>;
    auto kern = k_moment_pair<L, S, kPairH, kPairCtas, Step<S>>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, K::g_bytes) != cudaSuccess) return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, K::NT, K::g_bytes) != cudaSuccess || per_sm < 1)
        return 0;
    const int fit = per_sm * c.num_sms;
    return std::min(plan(c.nx, c.ny, c.nz, K::BX, K::BY, fit).nitems, fit);
}

template <class L, class S>
cudaError_t run_pair(const llb_ctx& c, const void* in, void* out, int zlo, int zhi, cudaStream_t stream, bool ghosts) {
    using K = PairTile<L, kPairH>;
    const int grid = c.tile_ctas > 0 ? c.tile_ctas : 1;
    const Sched sc = pair_plan(c, zhi - zlo, K::BX, K::BY, grid, ghosts);
    return launch_overlapped(k_moment_pair<L, S, kPairH, kPairCtas, Step<S>>, grid, K::NT, K::g_bytes, stream,
                             static_cast<const S*>(in), static_cast<S*>(out), c.lay,
                             Step<S>{coll_constants<L, S>(c.omega)}, sc, zlo, zhi - zlo, (int)(ghosts && c.lay.ghosts), static_cast<int*>(c.queue_dev));
}

}  // namespace mom
}  // namespace llb
