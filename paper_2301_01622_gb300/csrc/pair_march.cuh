// Pieces of the z-marching kernels that hold two nodes per thread
// (moment_pair.cuh, cg_pair.cuh).
//
// Thread (lane, w) owns the nodes (x, y) and (x, y + H) of a tile of 2H rows and
// does all its arithmetic and shared-memory accesses on the pair (float2: one
// packed instruction, one 8-byte access).  The exchange buffer holds "pair
// rows": pair row r is rows r and r + H of the tile, r = -1 .. H, so that a pair
// pulls along any direction with one aligned read.  Rows H - 1 and H border on
// both halves: the warps that own them write what crosses the seam a second
// time, into pair row -1 (second half) and pair row H (first half).
//
// Exchange.  Along an in-plane direction (cx, cy) the populations with c_z = -1,
// 0, 1 are c0 + zz - c1, c0, c0 + zz + c1 with
//   c0 = s + [cx] a_xx + [cy] a_yy + cx j_x + cy j_y + cx cy a_xy,
//   c1 = j_z + cx a_xz + cy a_yz, zz = a_zz (scaled moments of Col, below),
// so a node publishes c0 and c1 per direction and zz once, and the pull sums c0,
// c0 + zz and c1 separately before it forms the three planes.  The quantities are
// in units of the lattice's smallest weight and without the factors between the
// shells (D3Q19 1:2:12, D3Q27 1:4:16:64); the sums of the pull apply those in
// their multiply-adds.
#pragma once

#include "checked.cuh"
#include "lattice.cuh"
#include "layout.cuh"
#include "packed.cuh"

namespace llb {
namespace pk {

template <class L>
struct Shells;  // weights in units of the smallest: own column, in-plane axis, in-plane diagonal
template <>
struct Shells<D3Q19> {
    static constexpr bool corners = false;
    static constexpr double w = 1.0 / 36.0;
    static constexpr float own0 = 12.0f, axis0 = 2.0f, diag0 = 1.0f;  // c_z = 0
    static constexpr float own1 = 2.0f, axis1 = 1.0f;                 // c_z = +-1
};
template <>
struct Shells<D3Q27> {
    static constexpr bool corners = true;
    static constexpr double w = 1.0 / 216.0;
    static constexpr float own0 = 64.0f, axis0 = 16.0f, diag0 = 4.0f;
    static constexpr float own1 = 16.0f, axis1 = 4.0f;
};

// A collided node, in units of the smallest weight w: s = w (d - 1.5 tr A'),
// j = 3 w j, a_aa = 4.5 w A'_aa, a_ab = 9 w A'_ab, so that the population along
// c is s + sum of the a of c's components +- its j (Eq. (8)).
template <class V>
struct Col {
    V s, jx, jy, jz, xx, yy, zz, xy, xz, yz;
};

// s and j of a column with their constants in two parts.  Rounded to one float, 1/3 and
// 3 w are up to 3e-8 off: a fixed relative change of what a box conserves, which grows
// with the number of steps (256^3 D3Q19, 50 steps: 1.3e-9 of the mass from fl(1/3) alone).
template <class V>
__device__ __forceinline__ V col_s(V xx, V yy, V zz, V wd) {
    constexpr float hi = 1.0f / 3.0f, lo = (float)(1.0 / 3.0 - (double)hi);
    const V t = add(add(xx, yy), zz);
    return fma(-hi, t, fma(-lo, t, wd));
}
template <class V>
__device__ __forceinline__ V col_j(float hi, float lo, V j) {
    return fma(hi, j, mul(lo, j));
}

template <int CX, int CY, int CZ>
struct Dir {
    static constexpr int cx = CX, cy = CY, cz = CZ;
};

// Sums over the directions with one c_z of what an output node pulls from a
// source plane: sum g, sum g c_x, g c_y, g c_x c_x, g c_y c_y, g c_x c_y.
template <class V>
struct PlaneSum {
    V g, jx, jy, xx, yy, xy;
};

// In-plane directions (cx, cy) of the exchange: (1,0) (-1,0) (0,1) (0,-1) (1,1) (-1,-1) (1,-1) (-1,1).
__host__ __device__ constexpr int plane_dir(int cx, int cy) {
    return cy == 0 ? (cx > 0 ? 0 : 1) : cx == 0 ? (cy > 0 ? 2 : 3) : cx == cy ? (cx > 0 ? 4 : 5) : cx > 0 ? 6 : 7;
}

// Call put(Dir, c0, c1) for every in-plane direction with want(cx, cy).
template <class Want, class Put>
__device__ __forceinline__ void emit_plane(const Col<float2>& c, Want want, Put put) {
    const float2 ex = add(c.s, c.xx), ey = add(c.s, c.yy), exy = add(ex, c.yy);
    const float2 zp = add(c.jz, c.xz), zm = sub(c.jz, c.xz);
    const float2 u = add(exy, c.xy), v = sub(exy, c.xy), p = add(c.jx, c.jy), m = sub(c.jx, c.jy);
    auto one = [&](auto d, float2 c0, float2 c1) {
        using D = decltype(d);
        if (want(D::cx, D::cy)) put(d, c0, c1);
    };
    one(Dir<1, 0, 0>{}, add(ex, c.jx), zp);
    one(Dir<-1, 0, 0>{}, sub(ex, c.jx), zm);
    one(Dir<0, 1, 0>{}, add(ey, c.jy), add(c.jz, c.yz));
    one(Dir<0, -1, 0>{}, sub(ey, c.jy), sub(c.jz, c.yz));
    one(Dir<1, 1, 0>{}, add(u, p), add(zp, c.yz));
    one(Dir<-1, -1, 0>{}, sub(u, p), sub(zm, c.yz));
    one(Dir<1, -1, 0>{}, add(v, m), sub(zp, c.yz));
    one(Dir<-1, 1, 0>{}, sub(v, m), add(zm, c.yz));
}

// Sums over the eight neighbours of one published quantity, in the moments a
// plane accumulates (shell factors own : axis : diag; no diagonals if !D).
template <bool D>
__device__ __forceinline__ PlaneSum<float2> plane_sum(float own, float axis, float diag, float2 o, float2 ax,
                                                          float2 bx, float2 ay, float2 by, float2 pp, float2 mm,
                                                          float2 pm, float2 mp) {
    PlaneSum<float2> r;
    const float2 sx = add(ax, bx), dx = sub(ax, bx), sy = add(ay, by), dy = sub(ay, by);
    if constexpr (D) {
        const float2 a = add(pp, mm), b = add(pm, mp), c = sub(pp, mm), e = sub(pm, mp);
        const float2 sd = add(a, b);
        r.xx = fma(axis, sx, sd);
        r.yy = fma(axis, sy, sd);
        r.jx = fma(axis, dx, add(c, e));
        r.jy = fma(axis, dy, sub(c, e));
        r.xy = sub(a, b);
        r.g = fma(own, o, fma(axis, add(sx, sy), sd));
    } else {
        r.xx = sx;
        r.yy = sy;
        r.jx = dx;
        r.jy = dy;
        r.g = fma(own, o, add(sx, sy));
    }
    return r;
}

// Barrier of N threads of the CTA, reached by its warps at different places of the code.
template <int ID, int N>
__device__ __forceinline__ void bar_sync() {
    asm volatile("barrier.cta.sync.aligned %0, %1;" ::"n"(ID), "n"(N) : "memory");
}

}  // namespace pk
}  // namespace llb
