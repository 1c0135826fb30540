// Two-component moment-only step, FP32, two nodes per thread (pair_march.cuh).
//
// Same step as cg_kernel.cuh (its header has the equations).  That kernel
// executed 926 thread-instructions per node on D3Q27 and was bound by them; this
// one does less per node in four ways.
//   * Arithmetic and exchange on pairs of nodes.
//   * Loads and stores by TMA: the state is field-major, and a thread that loads and
//     stores its two nodes itself spends about five instructions per access on
//     addresses, 48 accesses per plane.
//   * The gradient of phi is a running sum: of each plane only the in-plane
//     differences and sums (9 reads) are taken, once, and combined with those of
//     the two planes before (kept in registers) instead of 26 reads of three planes.
//   * The colour populations h1'_i = (rho1/rho)(w_i + g'_i) + e w_i (c_i.n)/|c_i|
//     are not exchanged: a node publishes rho1/rho and e n once, and the pull forms
//     the sums of h1' from them and the g' it reads anyway.
//
// A CTA is H tile warps and a halo warp for the rows around the tile.  A warp
// holds 32 columns: the outputs are the inner 28, the next column on either side
// is collided for its populations only and the outermost for its phi only.  (A
// tile of 32 outputs with its side columns loaded apart was slower: those loads
// touch one sector of a line per lane, and cost the load pipe as much as the
// whole tile's.)  The rows above and below are doubled in the exchange (one copy for
// every other plane), so that the halo warp publishes plane s + 1 while the tile
// warps still pull plane s.
#pragma once

#include <algorithm>

#include "cg_kernel.cuh"
#include "cg_stages.cuh"
#include "overlap.cuh"
#include "pair_march.cuh"
#include "tma.cuh"

namespace llb {
namespace cg {

// Constants of the scaled collision: w = the smallest weight.
struct PairK {
    float ka, kc, ko;          // 4.5 w (1 - omega), 9 w (1 - omega), 4.5 w omega
    float w, w2, wj, wj2;      // w and 3 w, each with what rounding it left
    float kg, bw, kf;          // 0.5 w A_s, beta w, 9 w (1 - omega / 2)
    float A_h, g_min, g_nci, eps2;
    int h_c;
};

template <class L>
PairK pair_constants(const llb_ctx& c) {
    const double w = pk::Shells<L>::w, om = c.omega;
    PairK k;
    k.ka = (float)(4.5 * w * (1.0 - om));
    k.kc = (float)(9.0 * w * (1.0 - om));
    k.ko = (float)(4.5 * w * om);
    k.w = (float)w;
    k.w2 = (float)(w - (double)k.w);
    k.wj = (float)(3.0 * w);
    k.wj2 = (float)(3.0 * w - (double)k.wj);
    k.kg = (float)(0.5 * w * c.params.A_s);
    k.bw = (float)(c.params.beta * w);
    k.kf = (float)(9.0 * w * (1.0 - 0.5 * om));
    k.A_h = (float)c.params.A_h;
    k.eps2 = (float)(c.params.grad_eps * c.params.grad_eps);
    k.g_min = c.params.grad_eps > 0.0 ? 0.0f : (float)c.params.g_min;  // smooth norm: a normal everywhere
    k.g_nci = (float)kGNci;
    k.h_c = c.params.h_c;
    return k;
}

// In-plane terms of the gradient of phi around a node, and their running
// combination over three planes: G = unit * (gx, gy, gz).
//   D3Q27 (product weights): a = d_x (4, 1, 1 over y), b likewise, c = 16, 4, 1 sum;
//     g_x = a(s-1) + 4 a(s) + a(s+1), g_z = c(s+1) - c(s-1), unit = 3 / 216
//   D3Q19: a = d_x at the node's row, a1 = 2 a + d_x of the rows beside it;
//     g_x = a(s-1) + a1(s) + a(s+1), c = 2 phi + the four neighbours, unit = 3 / 36
template <class L>
struct PhiGrad {
    static constexpr bool kC = pk::Shells<L>::corners;
    static constexpr float unit = (float)(3.0 * pk::Shells<L>::w);
    float2 am, ac, a1, bm, bc, b1, cm, cc;

    // p(dy, dx): phi of plane s + 1 around the node; returns the gradient at plane s.
    template <class P>
    __device__ __forceinline__ void advance(P p, float2& gx, float2& gy, float2& gz) {
        using namespace pk;
        const float2 nw = p(-1, -1), nn = p(-1, 0), ne = p(-1, 1), ww = p(0, -1), oo = p(0, 0), ee = p(0, 1),
                     sw = p(1, -1), ss = p(1, 0), se = p(1, 1);
        const float2 dx0 = sub(ee, ww), dxr = add(sub(ne, nw), sub(se, sw));
        const float2 dy0 = sub(ss, nn), dyr = add(sub(sw, nw), sub(se, ne));
        const float2 four = add(add(ee, ww), add(ss, nn));
        float2 an, bn, cn;
        if constexpr (kC) {
            an = fma(4.0f, dx0, dxr);
            bn = fma(4.0f, dy0, dyr);
            cn = fma(16.0f, oo, fma(4.0f, four, add(add(nw, ne), add(sw, se))));
            gx = fma(4.0f, ac, add(am, an));
            gy = fma(4.0f, bc, add(bm, bn));
        } else {
            an = dx0;
            bn = dy0;
            cn = fma(2.0f, oo, four);
            gx = add(a1, add(am, an));
            gy = add(b1, add(bm, bn));
            a1 = fma(2.0f, dx0, dxr);
            b1 = fma(2.0f, dy0, dyr);
        }
        gz = sub(cn, cm);
        gx = mul(unit, gx);
        gy = mul(unit, gy);
        gz = mul(unit, gz);
        am = ac;
        ac = an;
        bm = bc;
        bc = bn;
        cm = cc;
        cc = cn;
    }
};

// Collided pair: the scaled moments, rho1 / rho and w e n.
struct Src {
    pk::Col<float2> c;
    float2 r1, ex, ey, ez;
};

// probe(want, n_out, phi0): the nodes of the pair (bits of want) in near contact.
template <class Probe>
__device__ __forceinline__ Src collide_pair(float2 r1, float2 d, const float2* m, float2 gx, float2 gy, float2 gz,
                                            const PairK& k, Probe probe) {
    using namespace pk;
    const float2 g2 = add(fma(gx, gx, fma(gy, gy, mul(gz, gz))), make_float2(k.eps2, k.eps2));
    float2 ig = make_float2(rsqrt_fast(fmaxf(g2.x, 1e-35f)), rsqrt_fast(fmaxf(g2.y, 1e-35f)));
    const float2 gn = mul(g2, ig);
    if (!(gn.x >= k.g_min)) ig.x = 0.0f;
    if (!(gn.y >= k.g_min)) ig.y = 0.0f;
    // 1 / rho, refined: rho1 is carried by rho1 / rho and sums of it with the weights, so what
    // the approximation or a weight is off by adds up from step to step (w2 for the same reason).
    // Error of 384 x 192 x 192 D3Q27 droplets after 30 steps against 64 bits, 2-norm, six inputs:
    // 3.6 to 6.2e-8 without the three, 2.3 to 3.2e-8 with them; 0.7 % of the step.
    const float2 one = make_float2(1.0f, 1.0f), r0 = rcp1p(1.0f, d);
    const float2 rinv = fma(r0, fma(sub(make_float2(-1.0f, -1.0f), d), r0, one), r0);
    Src s;
    s.r1 = mul(r1, rinv);
    // near-contact detector on the interface band
    int near = 0;
    if (k.A_h != 0.0f) {
        const int want = (gn.x >= k.g_nci ? 1 : 0) | (gn.y >= k.g_nci ? 2 : 0);
        if (want) {
            const float2 o = mul(-1.0f, ig);
            near = probe(want, mul(o, gx), mul(o, gy), mul(o, gz), fma(2.0f, s.r1, make_float2(-1.0f, -1.0f)));
        }
    }
    const float2 jx = m[0], jy = m[1], jz = m[2];
    auto collide = [&](float2 hx, float2 hy, float2 hz) {
        const float2 r = mul(k.ko, rinv), t = mul(k.kg, ig);
        const float2 ox = mul(r, hx), oy = mul(r, hy), oz = mul(r, hz);
        const float2 tx = mul(t, gx), ty = mul(t, gy), tz = mul(t, gz);
        s.c.xx = fma(tx, gx, fma(ox, hx, mul(k.ka, m[3])));
        s.c.yy = fma(ty, gy, fma(oy, hy, mul(k.ka, m[4])));
        s.c.zz = fma(tz, gz, fma(oz, hz, mul(k.ka, m[5])));
        const float2 ox2 = add(ox, ox), oy2 = add(oy, oy), tx2 = add(tx, tx), ty2 = add(ty, ty);
        s.c.xy = fma(tx2, gy, fma(ox2, hy, mul(k.kc, m[6])));
        s.c.xz = fma(tx2, gz, fma(ox2, hz, mul(k.kc, m[7])));
        s.c.yz = fma(ty2, gz, fma(oy2, hz, mul(k.kc, m[8])));
    };
    if (near) {  // F = A_h G on the nodes in near contact, u_F = (j + F / 2) / rho
        const float2 f = make_float2(near & 1 ? k.A_h : 0.0f, near & 2 ? k.A_h : 0.0f);
        const float2 fx = mul(f, gx), fy = mul(f, gy), fz = mul(f, gz);
        const float2 hx = fma(0.5f, fx, jx), hy = fma(0.5f, fy, jy), hz = fma(0.5f, fz, jz);
        collide(hx, hy, hz);
        const float2 u = mul(k.kf, rinv), ux = mul(u, hx), uy = mul(u, hy), uz = mul(u, hz);
        s.c.xx = fma(ux, fx, s.c.xx);
        s.c.yy = fma(uy, fy, s.c.yy);
        s.c.zz = fma(uz, fz, s.c.zz);
        s.c.xy = fma(ux, fy, fma(uy, fx, s.c.xy));
        s.c.xz = fma(ux, fz, fma(uz, fx, s.c.xz));
        s.c.yz = fma(uy, fz, fma(uz, fy, s.c.yz));
        s.c.jx = col_j(k.wj, k.wj2, add(jx, fx));
        s.c.jy = col_j(k.wj, k.wj2, add(jy, fy));
        s.c.jz = col_j(k.wj, k.wj2, add(jz, fz));
    } else {
        collide(jx, jy, jz);
        s.c.jx = col_j(k.wj, k.wj2, jx);
        s.c.jy = col_j(k.wj, k.wj2, jy);
        s.c.jz = col_j(k.wj, k.wj2, jz);
    }
    s.c.s = col_s(s.c.xx, s.c.yy, s.c.zz, mul(k.w, d));
    // e = beta rho1 rho2 / rho
    const float2 rho2 = add(sub(one, r1), d);
    const float2 e = mul(mul(mul(k.bw, s.r1), rho2), ig);
    s.ex = mul(e, gx);
    s.ey = mul(e, gy);
    s.ez = mul(e, gz);
    return s;
}

template <class L, int H_>
struct CgTile {
    static constexpr int W = 32, BX = W - 4, H = H_, BY = 2 * H_;
    static constexpr int NT = W * (H + 1);               // H tile warps and the halo warp
    // pair rows 0 .. H-1, two copies of the row above and two of the row below
    static constexpr int HN = W * (H + 4);
    static constexpr int PN = W * (H + 4);               // phi: pair rows -2 .. H+1
    static constexpr bool kC = pk::Shells<L>::corners;
    static constexpr int N4 = kC ? 8 : 4, N2 = kC ? 0 : 4;  // directions with (c0, c1), with c0 only
    // staged boxes: columns x0-4 .. x0+31; (rho1, d) rows -2 .. BY+1, four planes;
    // the other nine fields rows -1 .. BY, two planes; results: columns x0 .. x0+27
    static constexpr int SX = 36, RR = BY + 4, RM = BY + 2;
    static constexpr int RF = RR * SX, MF = RM * SX, OF = BY * BX;  // elements of one field
    static constexpr int up128(int b) { return (b + 127) / 128 * 128; }
    static constexpr int R_BYTES = 2 * RF * 4, M_BYTES = 9 * MF * 4, O_BYTES = 11 * OF * 4;
    static constexpr int R_SLOT = up128(R_BYTES), M_SLOT = up128(M_BYTES);
    static constexpr int R_OFF = 0, M_OFF = R_OFF + 4 * R_SLOT, O_OFF = M_OFF + 2 * M_SLOT;
    static constexpr int G_OFF = O_OFF + up128(O_BYTES);
    static constexpr int G_BYTES = HN * (16 * (N4 + 2) + 8 * (N2 + 1)) + 2 * 8 * PN;
    static constexpr int BAR_OFF = G_OFF + G_BYTES;
    static constexpr int smem_bytes = BAR_OFF + 16 + 128;  // two mbarriers; slack to align the base to 128 bytes
    static_assert(BX % 4 == 0, "box starts on 16-byte boundaries");
};

// Near contact of the pair (x, y0), (x, y1) in plane z: bit 0 / 1 of the result is
// set if phi at a probe node, k = 1 .. h_c along n_out = (ax, ay, az), exceeds its
// own phi0 by kPhiRise (want: bits to test).  The probes of both nodes are loaded
// three at a time, so that the step waits for memory once and not per probe; out
// of line, off the path of the nodes away from interfaces.
static __device__ __noinline__ int near_contact(const float* r1, const float* dd, int nx, int ny, int nz, int px,
                                                size_t plane, int x, int y0, int y1, int z, int h_c, int want,
                                                float2 ax, float2 ay, float2 az, float2 phi0) {
    // r1, dd: the fields at node (0, 0, 0); a box of at least 8 nodes wraps a probe at most once
    auto wrap = [](int v, int n) { return n >= 8 ? wrap_idx(v, n) : pmod2(v, n); };
    int got = 0;
#pragma unroll 1
    for (int todo = want; todo; todo &= todo - 1) {  // mostly one round: few lanes have both nodes on an interface
        const bool hi = !(todo & 1);
        const float bx = hi ? ax.y : ax.x, by = hi ? ay.y : ay.x, bz = hi ? az.y : az.x;
        const float t = (hi ? phi0.y : phi0.x) + (1.0f + (float)kPhiRise);
        const int y = hi ? y1 : y0;
        bool near = false;
#pragma unroll 1
        for (int q0 = 1; q0 <= h_c && !near; q0 += 3) {
            float r[3], d[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float q = (float)min(q0 + j, h_c);
                const int gx = wrap(x + __float2int_rn(q * bx), nx), gy = wrap(y + __float2int_rn(q * by), ny);
                const int gz = wrap(z + __float2int_rn(q * bz), nz);
                const size_t i = gz * plane + (unsigned)(gy * px + gx);
                const bool in_range = LLB_IN(i + 2 * px + kGhostX, plane * nz, kChkProbe);
                r[j] = in_range ? load_dep(r1 + i) : 0.0f;
                d[j] = in_range ? load_dep(dd + i) : 0.0f;
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) near |= 2.0f * r[j] > t * (1.0f + d[j]);  // phi = 2 rho1 / rho - 1 > phi0 + rise
        }
        if (near) got |= hi ? 2 : 1;
    }
    return got;
}

// Bound of a wait in cycles, and bytes that a barrier is armed for beyond those its copies
// deliver (fault injection: 0 in normal use).
struct WaitK {
    long long budget;
    int extra_tx;
};

// State that a CTA carries from item to item.
struct March {
    int par = 0;       // plane parity of the doubled exchange rows
    unsigned n = 0;    // staged groups waited for so far
    bool dead = false; // a wait gave up: no more waits or loads, the rest of the work is done on stale data
};

// One work item (z-chunk of one tile); arguments as cg_item.
//
// Staging.  Group n, waited for at the start of the step of source plane s, is
// the moments of plane s and (rho1, d) of plane s + 2 (the plane whose phi that
// step publishes); it is loaded two steps ahead, once the slots it overwrites
// have been read.
template <class L, int H>
__device__ __forceinline__ void cg_pair_item(const float* in, float* out, const CgMaps* __restrict__ maps,
                                             const Layout& lay, const PairK& k, const Sched2& sc, int it, int zlo,
                                             int nzr, March& st, int* err, const WaitK& wk) {
    using namespace pk;
    using C = CgTile<L, H>;
    using SH = Shells<L>;
    constexpr bool kC = C::kC;
    constexpr int W = C::W, BX = C::BX, BY = C::BY, HN = C::HN, PN = C::PN;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* const base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    float4* const G4 = reinterpret_cast<float4*>(base + C::G_OFF);  // (c0 lo, c0 hi, c1 lo, c1 hi) per direction
    float4* const B1 = G4 + C::N4 * HN;                             // (rho1/rho lo, hi, zz lo, hi)
    float4* const B2 = B1 + HN;                                     // (w e n_x lo, hi, w e n_y lo, hi)
    float2* const BZ = reinterpret_cast<float2*>(B2 + HN);          // w e n_z
    float2* const G2 = BZ + HN;                                     // c0 of the diagonals (D3Q19)
    float2* const PH = G2 + C::N2 * HN;                             // two planes of phi
    auto f4 = [](float4* p) { return reinterpret_cast<float*>(p); };
    auto f2 = [](float2* p) { return reinterpret_cast<float*>(p); };
    const uint32_t bar = smem_u32(base + C::BAR_OFF);

    const int nx = lay.nx, ny = lay.ny, nz = lay.nz;
    const size_t fs = lay.fs, plane = (size_t)lay.px * lay.py;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int chunk = it / sc.ntiles, tile = it - chunk * sc.ntiles;
    const int x0 = (tile % sc.ncx) * BX, y0 = (tile / sc.ncx) * BY;
    const int za = zlo + chunk * sc.zc, zb = min(zlo + nzr, za + sc.zc);
    const int ox = x0 - 2 + lane;  // column of this lane: column lane + 2 of the staged boxes
    auto phi_pair = [&](float2 r1, float2 d) {
        return pk::fma(2.0f, pk::mul(r1, rcp1p(1.0f, d)), make_float2(-1.0f, -1.0f));
    };
    int zs = pmod2(za - 4, nz);  // plane s, wrapped
    const float* const in00 = in + lay.at(0, 0, 0);
    const float2 zero = make_float2(0.0f, 0.0f);
    const int lf = max(lane - 1, 0), rt = min(lane + 1, W - 1);
    PhiGrad<L> gr{zero, zero, zero, zero, zero, zero, zero, zero};
    int pb = 0;  // phi buffer of plane s + 1
    auto rd_slot = [&](unsigned n) { return reinterpret_cast<const float*>(base + C::R_OFF + (n & 3) * C::R_SLOT); };
    auto m_slot = [&](unsigned n) { return reinterpret_cast<const float*>(base + C::M_OFF + (n & 1) * C::M_SLOT); };
    // load the group of step s (one thread)
    auto stage = [&](int s, unsigned n) {
        const uint32_t b = bar + 8 * Stages::bar(n);
        const bool mom = s >= za - 1, rd = s < zb;
        mbar_arrive_expect_tx(b, (mom ? C::M_BYTES : 0) + (rd ? C::R_BYTES : 0) + wk.extra_tx);
        if (rd)
            tma_load_4d(smem_u32(base + C::R_OFF + (n & 3) * C::R_SLOT), &maps->rd, x0 - 4 + lay.xo, y0 - 2 + lay.yo,
                        pmod2(s + 2, nz), 0, b);
        if (mom)
            tma_load_4d(smem_u32(base + C::M_OFF + (n & 1) * C::M_SLOT), &maps->m, x0 - 4 + lay.xo, y0 - 1 + lay.yo,
                        pmod2(s, nz), 2, b);
    };
    // Items taken after a wait gave up are not computed from loaded data: their box reports
    // it too, whichever box the wait was for.
    if (st.dead) atomicExch(err, 3);

    // Wait for the group of step s.  After a wait that gave up, the thread that issues the
    // copies lets those in flight land (bounded) before it goes on: later the barriers'
    // phases no longer tell which they were, and a CTA must not end with copies on the way
    // into its shared memory.
    auto await = [&](int s) {
        if (st.dead || mbar_wait_bounded(bar + 8 * Stages::bar(st.n), Stages::parity(st.n), wk.budget)) return;
        atomicExch(err, 3);
        st.dead = true;
        if (w == H && lane == 0)
            for (unsigned q = st.n; q != Stages::in_flight_end(st.n, s, zb); ++q)
                mbar_wait_bounded(bar + 8 * Stages::bar(q), Stages::parity(q), kDrainBudget);
    };

    // The march of every warp: source planes s = za - 4 .. zb; the first three only
    // fill the pipeline of phi (plane s + 2 is published in step s, plane s + 1 read).
    // Barrier 1: the exchange of plane s and phi of plane s + 2 are published;
    // barrier 2: the tile warps have pulled plane s.
    if (w == H) {
        // ---- halo warp: the pair of the rows -1 and BY, the latter mirrored in y, and
        // phi of the rows -2 and BY + 1
        // the halo warp also issues the loads
        const int xw = pmod2(ox, nx), ya = pmod2(y0 - 1, ny), yb = pmod2(y0 + BY, ny);
        const int ra = C::SX + lane + 2, rb = (BY + 2) * C::SX + lane + 2;  // its two nodes in a staged field
        if (lane == 0 && !st.dead) {
            stage(za - 4, st.n);
            stage(za - 3, st.n + 1);
        }
#pragma unroll 1
        for (int s = za - 4;; ++s) {
            __syncwarp();
            await(s);
            float2 gx, gy, gz;
            const float* const P = f2(PH + pb * PN);
            gr.advance([&](int dy, int dx) {
                const int l = dx < 0 ? lf : dx > 0 ? rt : lane;
                return make_float2(P[2 * ((1 + dy) * W + l)], P[2 * ((H + 2 + dy) * W + l) + 1]);
            }, gx, gy, gz);
            if (s >= za - 1) {
                const float *R = rd_slot(st.n - 2), *M = m_slot(st.n);
                float2 m[9];
#pragma unroll
                for (int f = 0; f < 9; ++f) m[f] = make_float2(M[f * C::MF + ra - C::SX], M[f * C::MF + rb - C::SX]);
                Src c = collide_pair(make_float2(R[ra], R[rb]), make_float2(R[C::RF + ra], R[C::RF + rb]), m, gx, gy, gz, k, [&](int want, float2 a, float2 b, float2 e, float2 phi0) {
                    return near_contact(in00, in00 + fs, nx, ny, nz, lay.px, plane, xw, ya, yb, zs, k.h_c, want, a, b, e, phi0);
                });
                c.c.jy.y = -c.c.jy.y;
                c.c.xy.y = -c.c.xy.y;
                c.c.yz.y = -c.c.yz.y;
                const int nt = (H + st.par) * W + lane, nb = (H + 2 + st.par) * W + lane;
                emit_plane(c.c, [](int, int cy) { return cy == 1; }, [&](auto dd, float2 c0, float2 c1) {
                    using D = decltype(dd);
                    constexpr int kt = plane_dir(D::cx, 1), kb = plane_dir(D::cx, -1);
                    if constexpr (kC || D::cx == 0) {
                        f4(G4)[4 * (kt * HN + nt)] = c0.x;
                        f4(G4)[4 * (kt * HN + nt) + 2] = c1.x;
                        f4(G4)[4 * (kb * HN + nb) + 1] = c0.y;
                        f4(G4)[4 * (kb * HN + nb) + 3] = c1.y;
                    } else {
                        f2(G2)[2 * ((kt - 4) * HN + nt)] = c0.x;
                        f2(G2)[2 * ((kb - 4) * HN + nb) + 1] = c0.y;
                    }
                });
                f4(B1)[4 * nt] = c.r1.x;
                f4(B1)[4 * nt + 2] = c.c.zz.x;
                f4(B2)[4 * nt] = c.ex.x;
                f4(B2)[4 * nt + 2] = c.ey.x;
                f2(BZ)[2 * nt] = c.ez.x;
                f4(B1)[4 * nb + 1] = c.r1.y;
                f4(B1)[4 * nb + 3] = c.c.zz.y;
                f4(B2)[4 * nb + 1] = c.ex.y;
                f4(B2)[4 * nb + 3] = c.ey.y;
                f2(BZ)[2 * nb + 1] = c.ez.y;
            }
            if (s < zb) {
                const float* R = rd_slot(st.n);
                float* const Q = f2(PH + (pb ^ 1) * PN);
                const int r0 = ra - C::SX, r3 = rb + C::SX;  // the rows -2 and BY + 1
                const float2 p = phi_pair(make_float2(R[ra], R[rb]), make_float2(R[C::RF + ra], R[C::RF + rb]));
                const float2 p2 = phi_pair(make_float2(R[r0], R[r3]), make_float2(R[C::RF + r0], R[C::RF + r3]));
                Q[2 * (W + lane)] = p.x;
                Q[2 * ((H + 2) * W + lane) + 1] = p.y;
                Q[2 * lane] = p2.x;
                Q[2 * ((H + 3) * W + lane) + 1] = p2.y;
            }
            zs = zs + 1 == nz ? 0 : zs + 1;
            pb ^= 1;
            st.par ^= 1;
            ++st.n;
            bar_sync<1, C::NT>();
            if (lane == 0 && s + 2 <= zb && !st.dead) stage(s + 2, st.n + 1);
            if (s == zb) break;
        }
        return;
    }

    // ---- tile warp: pair row w
    const int oy = y0 + w;
    const bool ok_x = lane >= 2 && lane < 2 + BX && ox < nx;
    const bool ok_lo = ok_x && oy < ny, ok_hi = ok_x && oy + H < ny;
    const int xw = pmod2(ox, nx), y_lo = pmod2(oy, ny), y_hi = pmod2(oy + H, ny);
    const int n1 = w * W + lane, p1 = (w + 2) * W + lane;
    const int rr = (w + 2) * C::SX + lane + 2, mr = (w + 1) * C::SX + lane + 2;  // the first node in a staged field
    float* const O = reinterpret_cast<float*>(base + C::O_OFF) + w * BX + lane - 2;
    // Periodic ghost copies: in a box at least 16 wide a node has at most one copy in
    // x and one in y; narrower boxes take the general form.
    const bool narrow_box = nx < 2 * kGhostX;
    const int gdx = ox < kGhostX ? nx : ox >= nx - kGhostX ? -nx : 0;
    auto row_copy = [&](int y) { return y < lay.yo ? ny * lay.px : y >= ny - lay.yo ? -ny * lay.px : 0; };
    const size_t o_lo = ok_lo ? lay.at(ox, oy, 0) : 0, o_hi = ok_hi ? lay.at(ox, oy + H, 0) : 0;
    // rolling sums of the plane ahead of the source plane (P) and of the source
    // plane (A; zg, zx, zy: the c_z moments of its c_z = +1 pulls).  Those of rho1 (Ph; Ah, Bh:
    // c_z = 0 and +1) stay apart until the last plane: rho1 is of order one and two roundings at
    // that size in every step, always the same way where the fluid is uniform, showed
    PlaneSum<float2> P{zero, zero, zero, zero, zero, zero}, A{zero, zero, zero, zero, zero, zero};
    float2 zg = zero, zx = zero, zy = zero, Ph = zero, Ah = zero, Bh = zero;

#pragma unroll 1
    for (int s = za - 4;; ++s) {
        await(s);
        float2 gx, gy, gz;
        {
            const float2* const Pp = PH + pb * PN + p1 - lane;
            gr.advance([&](int dy, int dx) { return Pp[dy * W + (dx < 0 ? lf : dx > 0 ? rt : lane)]; }, gx, gy, gz);
        }
        const bool work = s >= za - 1;
        float2 own_s = zero, own_z = zero;
        if (work) {
            const float *R = rd_slot(st.n - 2) + rr, *M = m_slot(st.n) + mr;
            float2 m[9];
#pragma unroll
            for (int f = 0; f < 9; ++f) m[f] = make_float2(M[f * C::MF], M[f * C::MF + H * C::SX]);
            const Src c = collide_pair(make_float2(R[0], R[H * C::SX]), make_float2(R[C::RF], R[C::RF + H * C::SX]), m, gx, gy, gz, k, [&](int want, float2 a, float2 b, float2 e, float2 phi0) {
                return near_contact(in00, in00 + fs, nx, ny, nz, lay.px, plane, xw, y_lo, y_hi, zs, k.h_c, want, a, b, e, phi0);
            });
            own_s = c.c.s;
            own_z = c.c.jz;
            if (LLB_IN(n1, HN, kChkPublish)) {
                emit_plane(c.c, [](int, int) { return true; }, [&](auto dd, float2 c0, float2 c1) {
                    using D = decltype(dd);
                    constexpr int kk = plane_dir(D::cx, D::cy);
                    const int up = (H + st.par) * W + lane, dn = (H + 2 + st.par) * W + lane;
                    if constexpr (kk < C::N4) {
                        G4[kk * HN + n1] = make_float4(c0.x, c0.y, c1.x, c1.y);
                        if (D::cy > 0 && w == H - 1) {
                            f4(G4)[4 * (kk * HN + up) + 1] = c0.x;
                            f4(G4)[4 * (kk * HN + up) + 3] = c1.x;
                        }
                        if (D::cy < 0 && w == 0) {
                            f4(G4)[4 * (kk * HN + dn)] = c0.y;
                            f4(G4)[4 * (kk * HN + dn) + 2] = c1.y;
                        }
                    } else {
                        G2[(kk - 4) * HN + n1] = c0;
                        if (D::cy > 0 && w == H - 1) f2(G2)[2 * ((kk - 4) * HN + up) + 1] = c0.x;
                        if (D::cy < 0 && w == 0) f2(G2)[2 * ((kk - 4) * HN + dn)] = c0.y;
                    }
                });
                B1[n1] = make_float4(c.r1.x, c.r1.y, c.c.zz.x, c.c.zz.y);
                B2[n1] = make_float4(c.ex.x, c.ex.y, c.ey.x, c.ey.y);
                BZ[n1] = c.ez;
                if (w == H - 1) {
                    const int up = (H + st.par) * W + lane;
                    f4(B1)[4 * up + 1] = c.r1.x;
                    f4(B1)[4 * up + 3] = c.c.zz.x;
                    f4(B2)[4 * up + 1] = c.ex.x;
                    f4(B2)[4 * up + 3] = c.ey.x;
                    f2(BZ)[2 * up + 1] = c.ez.x;
                }
                if (w == 0) {
                    const int dn = (H + 2 + st.par) * W + lane;
                    f4(B1)[4 * dn] = c.r1.y;
                    f4(B1)[4 * dn + 2] = c.c.zz.y;
                    f4(B2)[4 * dn] = c.ex.y;
                    f4(B2)[4 * dn + 2] = c.ey.y;
                    f2(BZ)[2 * dn] = c.ez.y;
                }
            }
        }
        if (s < zb) {
            const float* R = rd_slot(st.n) + rr;
            const float2 p = phi_pair(make_float2(R[0], R[H * C::SX]), make_float2(R[C::RF], R[C::RF + H * C::SX]));
            float2* const Q = PH + (pb ^ 1) * PN;
            if (LLB_IN(p1, PN, kChkPhi)) Q[p1] = p;
            if (w >= H - 2) f2(Q)[2 * (p1 - H * W) + 1] = p.x;
            if (w < 2) f2(Q)[2 * (p1 + H * W)] = p.y;
        }
        zs = zs + 1 == nz ? 0 : zs + 1;
        pb ^= 1;
        ++st.n;
        if (threadIdx.x == 0) bulk_wait_read();  // the results staged last step have been read
        bar_sync<1, C::NT>();
        if (work) {
            const int up = (w == 0 ? H + st.par : w - 1) * W, dn = (w == H - 1 ? H + 2 + st.par : w + 1) * W, mid = w * W;
            auto lo2 = [](float4 v) { return make_float2(v.x, v.y); };
            auto hi2 = [](float4 v) { return make_float2(v.z, v.w); };
            auto at = [&](int row, int col) { return LLB_IN(row + col, HN, kChkGather) ? row + col : 0; };
            const int nl = at(mid, lf), nr = at(mid, rt), nu = at(up, lane), nd = at(dn, lane);
            const int nul = at(up, lf), nur = at(up, rt), ndl = at(dn, lf), ndr = at(dn, rt);
            const float i2 = 0.70710678118654752440f, i3 = 0.57735026918962576451f;
            // Shell factors; those of D3Q27's c_z = 0 plane are 4 times the other planes' and applied last.
            constexpr float s0 = kC ? 4.0f : 1.0f, o0 = SH::own0 / s0, a0 = SH::axis0 / s0, o1 = SH::own1, a1 = SH::axis1;
            // h1' along c without its shell factor: r1 (w + g) + (c.E) / |c|, E = w e n; its sums
            // over the neighbours: r1 c0, r1 (c0 + zz), r1 c1 and the part without g'
            struct Nb {
                float2 c0, c1, t, r;
            };
            auto nb = [&](int kk, int n) {
                const float4 c = G4[kk * HN + n], b = B1[n];
                return Nb{lo2(c), hi2(c), add(lo2(c), hi2(b)), lo2(b)};
            };
            const Nb l = nb(0, nl), r = nb(1, nr), u = nb(2, nu), d = nb(3, nd);
            float2 h0 = fma(l.r, l.c0, fma(r.r, r.c0, fma(u.r, u.c0, mul(d.r, d.c0))));
            float2 ht = fma(l.r, l.t, fma(r.r, r.t, fma(u.r, u.t, mul(d.r, d.t))));
            float2 hc = fma(l.r, l.c1, fma(r.r, r.c1, fma(u.r, u.c1, mul(d.r, d.c1))));
            {
                const float2 R = col_j(k.w, k.w2, add(add(l.r, r.r), add(u.r, d.r)));
                const float2 T = add(sub(lo2(B2[nl]), lo2(B2[nr])), sub(hi2(B2[nu]), hi2(B2[nd])));
                const float2 Z = add(add(BZ[nl], BZ[nr]), add(BZ[nu], BZ[nd]));
                h0 = mul(a0, add(h0, add(R, T)));
                ht = mul(a1, add(ht, fma(i2, T, R)));
                hc = mul(a1, fma(i2, Z, hc));
            }
            PlaneSum<float2> q0, qt, qc;
            {
                const float4 e = B2[nul], f = B2[nur], g = B2[ndl], h = B2[ndr];
                const float2 T = add(add(sub(lo2(e), lo2(f)), sub(lo2(g), lo2(h))),
                                     sub(add(hi2(e), hi2(f)), add(hi2(g), hi2(h))));
                if constexpr (kC) {
                    const Nb pp = nb(4, nul), mm = nb(5, ndr), pm = nb(6, ndl), mp = nb(7, nur);
                    const float2 R = col_j(k.w, k.w2, add(add(pp.r, mm.r), add(pm.r, mp.r)));
                    const float2 Z = add(add(BZ[nul], BZ[nur]), add(BZ[ndl], BZ[ndr]));
                    h0 = fma(pp.r, pp.c0, fma(mm.r, mm.c0, fma(pm.r, pm.c0, fma(mp.r, mp.c0, h0))));
                    ht = fma(pp.r, pp.t, fma(mm.r, mm.t, fma(pm.r, pm.t, fma(mp.r, mp.t, ht))));
                    hc = fma(pp.r, pp.c1, fma(mm.r, mm.c1, fma(pm.r, pm.c1, fma(mp.r, mp.c1, hc))));
                    h0 = add(h0, fma(i2, T, R));
                    ht = add(ht, fma(i3, T, R));
                    hc = fma(i3, Z, hc);
                    qt = plane_sum<true>(o1, a1, 1.0f, add(own_s, hi2(B1[n1])), l.t, r.t, u.t, d.t, pp.t, mm.t, pm.t, mp.t);
                    qc = plane_sum<true>(o1, a1, 1.0f, own_z, l.c1, r.c1, u.c1, d.c1, pp.c1, mm.c1, pm.c1, mp.c1);
                    q0 = plane_sum<true>(o0, a0, 1.0f, own_s, l.c0, r.c0, u.c0, d.c0, pp.c0, mm.c0, pm.c0, mp.c0);
                } else {
                    const float2 pp = G2[nul], mm = G2[HN + ndr], pm = G2[2 * HN + ndl], mp = G2[3 * HN + nur];
                    const float2 rp = lo2(B1[nul]), rm = lo2(B1[ndr]), rq = lo2(B1[ndl]), rs = lo2(B1[nur]);
                    const float2 R = col_j(k.w, k.w2, add(add(rp, rm), add(rq, rs)));
                    h0 = fma(rp, pp, fma(rm, mm, fma(rq, pm, fma(rs, mp, h0))));
                    h0 = add(h0, fma(i2, T, R));
                    qt = plane_sum<false>(o1, a1, 1.0f, add(own_s, hi2(B1[n1])), l.t, r.t, u.t, d.t, zero, zero, zero, zero);
                    qc = plane_sum<false>(o1, a1, 1.0f, own_z, l.c1, r.c1, u.c1, d.c1, zero, zero, zero, zero);
                    q0 = plane_sum<true>(o0, a0, 1.0f, own_s, l.c0, r.c0, u.c0, d.c0, pp, mm, pm, mp);
                }
            }
            {  // own column
                const float4 v = B1[n1];
                const float2 rr = lo2(v), ws = add(own_s, make_float2(k.w, k.w));
                const float2 r0 = mul(o0, rr), r1 = mul(o1, rr);
                h0 = fma(r0, ws, fma(k.w2, r0, h0));
                ht = fma(r1, add(ws, hi2(v)), fma(k.w2, r1, ht));
                hc = fma(o1, fma(rr, own_z, BZ[n1]), hc);
            }
            {  // plane s - 1 is complete with the c_z = -1 pulls, qt - qc
                float2 v[11];
                const float third = (float)kCs2;
                const float2 g = sub(qt.g, qc.g), jx = sub(qt.jx, qc.jx), jy = sub(qt.jy, qc.jy);
                v[0] = fma(s0, Ah, add(Bh, sub(ht, hc)));
                v[1] = add(A.g, g);
                v[2] = add(A.jx, jx);
                v[3] = add(A.jy, jy);
                v[4] = sub(zg, g);
                v[5] = fma(-third, v[1], add(A.xx, sub(qt.xx, qc.xx)));
                v[6] = fma(-third, v[1], add(A.yy, sub(qt.yy, qc.yy)));
                v[7] = fma(-third, v[1], add(zg, g));
                v[8] = kC ? add(A.xy, sub(qt.xy, qc.xy)) : A.xy;
                v[9] = sub(zx, jx);
                v[10] = sub(zy, jy);
                if (s > za) {
                    if (lane >= 2 && lane < 2 + BX) {
#pragma unroll
                        for (int f = 0; f < 11; ++f) {
                            O[f * C::OF] = v[f].x;
                            O[f * C::OF + H * BX] = v[f].y;
                        }
                    }
                    fence_proxy_async();
                    const size_t zw = (size_t)(s - 1) * plane;
                    auto store = [&](size_t o, int dd, bool hi) {
                        if (!LLB_IN((long long)(zw + o) + dd, fs, kChkGhost)) return;
                        float* p = out + (zw + o) + dd;
#pragma unroll
                        for (int f = 0; f < 11; ++f, p += fs) *p = hi ? v[f].y : v[f].x;
                    };
                    if (!narrow_box) {
                        if (gdx) {
                            if (ok_lo) store(o_lo, gdx, false);
                            if (ok_hi) store(o_hi, gdx, true);
                        }
                        const int gl = row_copy(oy), gh = row_copy(oy + H);
                        if (gl && ok_lo) {
                            store(o_lo, gl, false);
                            if (gdx) store(o_lo, gl + gdx, false);
                        }
                        if (gh && ok_hi) {
                            store(o_hi, gh, true);
                            if (gdx) store(o_hi, gh + gdx, true);
                        }
                    } else {
#pragma unroll 1
                        for (int hi = 0; hi < 2; ++hi) {
                            if (hi ? !ok_hi : !ok_lo) continue;
                            Mom<float> mm;
                            mm.d = hi ? v[1].y : v[1].x;
                            mm.jx = hi ? v[2].y : v[2].x;
                            mm.jy = hi ? v[3].y : v[3].x;
                            mm.jz = hi ? v[4].y : v[4].x;
                            mm.axx = hi ? v[5].y : v[5].x;
                            mm.ayy = hi ? v[6].y : v[6].x;
                            mm.azz = hi ? v[7].y : v[7].x;
                            mm.axy = hi ? v[8].y : v[8].x;
                            mm.axz = hi ? v[9].y : v[9].x;
                            mm.ayz = hi ? v[10].y : v[10].x;
                            store_node2(out, lay, ox, oy + hi * H, s - 1, hi ? v[0].y : v[0].x, mm);
                        }
                    }
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
            Ah = h0;
            Bh = Ph;
            P.g = add(qt.g, qc.g);
            P.jx = add(qt.jx, qc.jx);
            P.jy = add(qt.jy, qc.jy);
            P.xx = add(qt.xx, qc.xx);
            P.yy = add(qt.yy, qc.yy);
            if constexpr (kC) P.xy = add(qt.xy, qc.xy);
            Ph = add(ht, hc);
            bar_sync<2, 32 * H>();
            if (threadIdx.x == 0 && s > za) {
                tma_store_4d(&maps->out, smem_u32(base + C::O_OFF), x0, y0, s - 1, 0);
                bulk_commit();
            }
        }
        st.par ^= 1;
        if (s == zb) break;
    }
}

// Staging barriers up; every warp of the CTA.
template <class C>
__device__ __forceinline__ void cg_pair_begin() {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = smem_u32(smem_raw), bar = base + ((128 - (base & 127)) & 127) + C::BAR_OFF;
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 8, 1);
        fence_barrier_init();
    }
    __syncthreads();
}

template <class L, int H, int MINB>
__global__ void __launch_bounds__(32 * (H + 1), MINB)
    k_cg_pair(const float* in, float* out, const __grid_constant__ CgMaps maps, Layout lay,
              PairK k, Sched2 sc, int zlo, int nzr, int* err, int* queue, WaitK wk) {
    using C = CgTile<L, H>;
    cg_pair_begin<C>();
    March st;
    // Items from a queue (queue[0]: next item, queue[1]: CTAs done): those that hold an
    // interface take longer.  The last CTA to leave resets it for the next launch.
    __shared__ int s_it;
    dep_wait();
    for (;;) {
        if (threadIdx.x == 0) s_it = atomicAdd(queue, 1);
        __syncthreads();
        const int it = s_it;
        __syncthreads();
        if (it >= sc.nitems) break;
        cg_pair_item<L, H>(in, out, &maps, lay, k, sc, it, zlo, nzr, st, err, wk);
    }
    dep_launch();
    if (threadIdx.x == 0) bulk_wait();  // results out
    if (threadIdx.x == 0 && atomicAdd(queue + 1, 1) == (int)gridDim.x - 1) {
        queue[0] = 0;
        queue[1] = 0;
    }
}

// Batched ensemble, work queue as in k_cg_batch.  maps: one entry per box.
template <class L, int H, int MINB>
__global__ void __launch_bounds__(32 * (H + 1), MINB)
    k_cg_pair_batch(const BatchDom* __restrict__ doms, const CgMaps* __restrict__ maps, int ndom, int total, PairK k,
                    int* __restrict__ next, WaitK wk) {
    using C = CgTile<L, H>;
    __shared__ int s_it;
    cg_pair_begin<C>();
    March st;
    for (;;) {
        if (threadIdx.x == 0) s_it = atomicAdd(next, 1);
        __syncthreads();
        const int it = s_it;
        __syncthreads();
        if (it >= total) break;
        int lo = 0, hi = ndom - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (doms[mid].item_begin <= it) lo = mid;
            else hi = mid - 1;
        }
        const BatchDom d = doms[lo];
        const Sched2 sc{d.ncx, d.ntiles, d.zc, d.nitems};
        // the two threads that issue copies acquire the box's maps
        if (threadIdx.x == C::NT - 32) {
            acquire_tensormap(&maps[lo].rd);
            acquire_tensormap(&maps[lo].m);
        }
        if (threadIdx.x == 0) acquire_tensormap(&maps[lo].out);
        cg_pair_item<L, H>(static_cast<const float*>(d.in), static_cast<float*>(d.out), maps + lo, d.lay, k, sc,
                           it - d.item_begin, 0, d.lay.nz, st, d.err, wk);
    }
    if (threadIdx.x == 0) bulk_wait();  // results out
}

// Tiles of 28 x 10, two CTAs of six warps per SM (168 registers, no spills; 113 KB
// of shared memory each on D3Q27).  Measured on 384 x 192 x 192 D3Q27 with a droplet
// pair, 128^3 D3Q19 and 96^3 D3Q27 (A_h = 0): 459, 87, 45 us per step (464 on the first since
// the roundings of rho1 are kept small); one CTA of 12
// warps (28 x 22): 463, 92, 49 us; CTAs of four warps (28 x 6): 531, 86, 53 us; eight
// warps at 128 registers spill and lose 15 % and more.
constexpr int kPairH = 5, kPairCtas = 2;

// Tensor maps of a step from `in` to `out`.
inline bool cg_pair_maps(const llb_ctx& c, const void* in, void* out, CgMaps* m) {
    using C = CgTile<D3Q19, kPairH>;  // the boxes are those of either lattice
    const Layout& y = c.lay;
    const size_t row = (size_t)y.px * 4, plane = row * y.py, fs = y.fs * 4;
    const size_t all[4] = {(size_t)y.px, (size_t)y.py, (size_t)y.nz, 11}, inner[4] = {(size_t)y.nx, (size_t)y.ny, (size_t)y.nz, 11};
    const size_t strides[3] = {row, plane, fs};
    const int rd[4] = {C::SX, C::RR, 1, 2}, mo[4] = {C::SX, C::RM, 1, 9}, res[4] = {C::BX, C::BY, 1, 11};
    return encode_f32_map(const_cast<void*>(in), all, strides, rd, &m->rd) &&
           encode_f32_map(const_cast<void*>(in), all, strides, mo, &m->m) &&
           encode_f32_map(static_cast<float*>(out) + y.at(0, 0, 0), inner, strides, res, &m->out);
}

// device clock ~2 GHz: cycles per millisecond
inline WaitK wait_bounds(const llb_ctx& c) {
    return {(long long)c.params.wait_budget_ms * 2000000LL, (c.params.debug_flags & 1) ? 1 : 0};
}

// Chunk length of a box whose items go through the queue on `grid` CTAs.  A step
// of an item costs about its planes plus 3.5 to fill the pipeline.  Without near
// contact all items cost the same and fill whole rounds; with it those on an
// interface take up to twice as long, so the items are made short enough that the
// queue evens them out.
inline Sched2 cg_pair_plan(const llb_ctx& c, int nzr, int BX, int BY, int grid) {
    Sched2 s;
    s.ncx = (c.nx + BX - 1) / BX;
    s.ntiles = s.ncx * ((c.ny + BY - 1) / BY);
    double best = -1.0;
    for (int nch = 1; nch <= nzr; ++nch) {
        const int zc = (nzr + nch - 1) / nch, chunks = (nzr + zc - 1) / zc;
        const long long items = (long long)s.ntiles * chunks;
        if (items > (1LL << 30)) break;
        const double rounds = c.params.A_h != 0.0 ? (double)items / grid + 0.75 : (double)((items + grid - 1) / grid);
        const double cost = rounds * (zc + 3.5);
        if (best < 0.0 || cost < best) {
            best = cost;
            s.zc = zc;
            s.nitems = (int)items;
        }
    }
    return s;
}

// Persistent CTAs of `kern` that fit the chip, 0 if it cannot run.
template <class C, class K>
int cg_pair_fit(const llb_ctx& c, K kern) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::smem_bytes) != cudaSuccess) return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::NT, C::smem_bytes) != cudaSuccess) return 0;
    return per_sm * c.num_sms;
}

}  // namespace cg
}  // namespace llb
