// Pieces of the z-marching kernels that hold two nodes per thread (cg_pair.cuh).
//
// Thread (lane, w) owns the nodes (x, y) and (x, y + H) of a tile of 2H rows and
// does all its arithmetic and shared-memory accesses on the pair (float2: one
// packed instruction, one 8-byte access).  The exchange buffer holds "pair
// rows": pair row r is rows r and r + H of the tile, r = -1 .. H, so that a pair
// pulls along any direction with one aligned read.  Rows H - 1 and H border on
// both halves: the warps that own them write what crosses the seam a second
// time, into pair row -1 (second half) and pair row H (first half).
//
// Populations are exchanged in units of the lattice's smallest weight and
// without the factors between the shells (D3Q19 1:2:12, D3Q27 1:4:16:64); the
// sums of the pull apply those in their multiply-adds.
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

// Barrier of N threads of the CTA, reached by its warps at different places of the code.
template <int ID, int N>
__device__ __forceinline__ void bar_sync() {
    asm volatile("barrier.cta.sync.aligned %0, %1;" ::"n"(ID), "n"(N) : "memory");
}

}  // namespace pk
}  // namespace llb
