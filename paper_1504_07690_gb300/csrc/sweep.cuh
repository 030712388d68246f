// sweep.cuh - shared pieces of the kernels that sweep the planes of a grid along axis 0
// (stencil steps in recurrence.cu, the adjoint step in adjoint.cu).
//
// A CTA owns a T1 x T2 tile of axes 1 and 2 and a run of planes.  The adjoint step's planes
// (with their halo) go through a ring of shared-memory slots filled by asynchronous copies,
// PF planes ahead, so that the loads in flight take no registers.  The forward step keeps
// three planes of its element in registers and only the current one, with its halo, in
// shared memory (PF = 0: no ring).
#pragma once

#include "internal.h"

namespace ssm {

template <int T1_, int T2_, int PF_ = 0>
struct SweepTile {
    static constexpr int T1 = T1_, T2 = T2_, ROWS = T1 * T2, W2 = T2 + 2;
    static constexpr int H1 = T1 > 1 ? 1 : 0;             // halo along axis 1 (T1 = 1: the axis is inactive)
    static constexpr int HALO1 = 2 * H1 * T2;             // its rows
    static constexpr int HALO = HALO1 + 2 * T1;
    static constexpr int PLANE = (T1 + 2 * H1) * W2;      // rows of a staged plane
    static constexpr int PF = PF_, NSLOT = PF + 1;
};

// Coordinate q in [-1, ext] of an axis, or -1 where nothing is there.
__device__ __forceinline__ int axis_at(int q, int ext, bool per) {
    if (q >= 0 && q < ext) return q;
    if (!per || q > ext) return -1;
    return q < 0 ? ext - 1 : 0;
}

// 16 bytes global -> shared, asynchronously; ok = false: zeros, nothing is read.
template <typename V>
__device__ __forceinline__ void async16(V* dst, const V* src, bool ok) {
    static_assert(sizeof(V) == 16, "16-byte elements");
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Where in a staged plane a row of threads puts its element and its share of the halo:
// offsets in rows of the plane and coordinates relative to the tile.
template <typename ST>
struct SweepRow {
    int r1, r2;      // the row's place in the tile
    bool halo, ax1;  // the row also fetches a halo element: of an axis-1 side, else axis 2
    int h1, h2;      // its place
    __device__ explicit SweepRow(int r) {
        r1 = r / ST::T2;
        r2 = r % ST::T2;
        halo = r < ST::HALO;
        ax1 = r < ST::HALO1;
        const int k = ax1 ? r % ST::T2 : (r - ST::HALO1) % ST::T1;
        const bool hi = ax1 ? r >= ST::T2 : r - ST::HALO1 >= ST::T1;
        h1 = ax1 ? (hi ? ST::T1 : -1) : k;
        h2 = ax1 ? k : (hi ? ST::T2 : -1);
    }
    __device__ uint32_t own_at() const { return (uint32_t)(r1 + ST::H1) * ST::W2 + r2 + 1; }
    __device__ uint32_t halo_at() const { return halo ? (uint32_t)(h1 + ST::H1) * ST::W2 + h2 + 1 : 0; }
};

// Tiles and runs of a launch; nseg = 0 where a tiled sweep does not pay: a grid too thin
// for the tiles (more than a quarter of their rows past its edges) or of few planes.
struct SweepRuns {
    uint32_t nt1 = 0, nt2 = 0, planes = 0, nseg = 0;
};

// Runs of planes for about `want` CTAs over the launch (groups: CTAs per tile and run), at
// least min_planes planes each (a run reads one plane more at either end).
template <typename ST>
inline SweepRuns sweep_runs(uint32_t d0, uint32_t d1, uint32_t d2, uint64_t groups, uint64_t want,
                            uint32_t min_planes) {
    SweepRuns w;
    const uint64_t nt1 = (d1 + ST::T1 - 1) / ST::T1, nt2 = (d2 + ST::T2 - 1) / ST::T2;
    const uint64_t tiles = nt1 * nt2;
    if (d0 < 4 || 3 * tiles * ST::ROWS > 4 * (uint64_t)d1 * d2 || tiles * groups > 0x7fffffff) return w;
    uint64_t nseg = (want + tiles * groups - 1) / (tiles * groups);
    if (nseg > d0 / min_planes) nseg = d0 / min_planes;
    if (nseg > 65535) nseg = 65535;
    if (nseg < 1) nseg = 1;
    w.nt1 = (uint32_t)nt1;
    w.nt2 = (uint32_t)nt2;
    w.planes = (uint32_t)((d0 + nseg - 1) / nseg);
    w.nseg = (d0 + w.planes - 1) / w.planes;
    return w;
}

}  // namespace ssm
