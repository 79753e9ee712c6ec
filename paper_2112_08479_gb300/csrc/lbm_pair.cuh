// lbm_pair.cuh -- AA gather / scatter of the nodes x and x + 32 of a row by
// one thread: a warp owns a segment of 64 x-consecutive nodes, lane l the
// nodes l and 32 + l, so that every population row is moved as two contiguous
// 32-element requests per warp on any alignment, and the two nodes' values are
// the halves of one packed register pair for the collision (lbm_lanes.cuh).
//
// Sides.  For an opposite pair of directions (i, i + 1), i odd, an odd AA step
// of node n touches two elements (lbm_common.cuh):
//   P: slot i of node n + c_i          M: slot i + 1 of node n - c_i
// reads f_(i+1) from P and f_i from M, and writes f*_i to P and f*_(i+1) to M.
// Where the neighbour of a side lies beyond a wall, the side is the slot of
// the opposite direction of node n itself, for the read and for the write.
// An even step touches slot i (P) and slot i + 1 (M) of node n; it reads f_i
// from P and f_(i+1) from M and writes them crosswise.  Naming the population
// read from M f_i on even steps too therefore leaves one code for both
// parities: the nodes then see the mirrored velocity set c -> -c, and the
// collision gets -F.
//
// So a step is described by one element offset per side, the same for every
// lane of a row segment away from the x ends: PairTable holds them for the
// even step and, for odd steps, for each position of the row in y (periodic
// wrap) and z (walls or wrap).  Segments at the x ends (EDGE) resolve their
// first and last columns and the lanes beyond the row per lane.
#pragma once

#include <type_traits>

#include "lbm_internal.h"
#include "lbm_lanes.cuh"

namespace lbmgpu {

constexpr int PAIR_CLASSES = 17;   // the even step; odd: 1 + 4 (z position) + (y position)

// Element offsets from the node to the sides of the fluid (F opposite pairs)
// and of the scalar (G opposite pairs): [2 m] is side P of pair m, [2 m + 1]
// side M; formed modulo 2^32.  Arrays of 2^32 elements or more (WIDE,
// KParams::wide) hold them relative to the first of the pair's two rows, whose
// 64-bit base is the same for every thread: node and offset then make less than
// 2 N < 2^32.
template <int F, int G>
struct PairTable {
    unsigned f[PAIR_CLASSES][2 * F];
    unsigned g[PAIR_CLASSES][2 * G];
};

// Position of a coordinate: 0 inside, 1 first, 2 last, 3 both (extent 1).
__host__ __device__ constexpr int pair_pos(int c, int n) {
    return (c == 0 ? 1 : 0) + (c == n - 1 ? 2 : 0);
}

// Fills the sides of M opposite pairs of directions 1, 2, ... whose rows are
// direction - d0.
template <int M>
inline void pair_sides(const KParams& kp, int d0, unsigned (&o)[PAIR_CLASSES][2 * M]) {
    const long long N = kp.N;
    const bool pz = (kp.flags & LBM_FLAG_PERIODIC_Z) != 0;
    for (int cls = 0; cls < PAIR_CLASSES; ++cls) {
        const int yp = cls ? (cls - 1) % 4 : 0, zp = cls ? (cls - 1) / 4 : 0;
        for (int m = 0; m < M; ++m) {
            const int i = 2 * m + 1, row = kp.wide ? 0 : i - d0;   // of direction i
            for (int side = 0; side < 2; ++side) {
                const int s = side == 0 ? 1 : -1;   // P: n + c_i, M: n - c_i
                const long long own = (row + (side == 0 ? 0 : 1)) * N;
                const long long other = (row + (side == 0 ? 1 : 0)) * N;
                long long v = own;
                if (cls) {
                    const int cx = s * cx27(i), cy = s * cy27(i), cz = s * cz27(i);
                    const bool zlo = cz < 0 && (zp & 1), zhi = cz > 0 && (zp & 2);
                    const bool ylo = cy < 0 && (yp & 1), yhi = cy > 0 && (yp & 2);
                    if ((zlo || zhi) && !pz) {
                        v = other;
                    } else {
                        v += cx;
                        v += (long long)(cy + (ylo ? kp.ny : (yhi ? -kp.ny : 0))) * kp.nx;
                        v += (long long)(cz + (zlo ? kp.nz : (zhi ? -kp.nz : 0))) * kp.nxny;
                    }
                }
                o[cls][2 * m + side] = (unsigned)v;
            }
        }
    }
}

template <int F, int G>
inline void pair_table(const KParams& kp, int d0, PairTable<F, G>& t) {
    pair_sides<F>(kp, 0, t.f);
    pair_sides<G>(kp, d0, t.g);
}

// The context's copy (Sides), as the type it was filled with.
template <int F, int G>
inline PairTable<F, G>& pair_view(Sides& s) {
    static_assert(sizeof(PairTable<F, G>) <= sizeof s.bytes);
    return *reinterpret_cast<PairTable<F, G>*>(s.bytes);
}
template <int F, int G>
inline const PairTable<F, G>& pair_view(const Sides& s) {
    return pair_view<F, G>(const_cast<Sides&>(s));
}

// Warps of a block along x (of ns 64-node segments per row): as many, up to
// four, as leave the fewest idle.
inline int pair_warps(int ns) {
    if (ns <= 4) return ns;
    for (int w = 4; w > 2; --w)
        if (ns % w == 0) return w;
    return ns % 4 == 1 ? 3 : 4;
}

// The nodes of a thread.
struct PairNodes {
    unsigned n;          // node x; the other one is n + 32
    int x;
    bool odd;
    int zwall;           // 1: no plane below (a wall), 2: none above
    // node x + d, or the row's last node where x + d is beyond it
    __device__ __forceinline__ unsigned clamped(const KParams& kp, int d) const {
        return n + (unsigned)(min(x + d, kp.nx - 1) - x);
    }
};

__device__ __forceinline__ PairNodes pair_nodes(const KParams& kp, int x0, int y, int z, bool odd) {
    PairNodes pn;
    pn.x = x0 + (int)(threadIdx.x & 31);
    pn.n = (unsigned)z * kp.nxny + (unsigned)y * kp.nx + (unsigned)pn.x;
    pn.odd = odd;
    pn.zwall = (kp.flags & LBM_FLAG_PERIODIC_Z) ? 0 : pair_pos(z, kp.nz);
    return pn;
}

// Class of a row in the table.  The reduction over the warp (every lane has the
// same value) leaves it in a uniform register, so that the table is read by
// uniform loads: with a per-lane index the offsets took vector registers and
// spilled.
__device__ __forceinline__ int pair_class(const KParams& kp, bool odd, int y, int z) {
    const int c = odd ? 1 + 4 * pair_pos(z, kp.nz) + pair_pos(y, kp.ny) : 0;
    return (int)__reduce_max_sync(0xffffffffu, (unsigned)c);
}

// True when all 64 nodes of the segment at x0 exist and have both x neighbours
// inside the box.
__device__ __forceinline__ bool pair_inner(const KParams& kp, int x0) {
    return x0 >= 1 && x0 + 64 <= kp.nx - 1;
}

// Offset of a side for the node at x: the table's, except on odd steps where
// the side's x neighbour leaves the box at this node: the own slot of the
// opposite direction (row `other`) at a wall (as the table has it already
// where the side meets a z wall), the wrapped column with periodic ends.
// dx, dz: the side's displacement.
__host__ __device__ __forceinline__ unsigned pair_edge(const KParams& kp, const PairNodes& pn,
                                                       int x, unsigned off, unsigned other, int dx,
                                                       int dz) {
    // (selects, no branches: the loads that follow must not wait for each other)
    const bool turned = (dz < 0 && (pn.zwall & 1)) || (dz > 0 && (pn.zwall & 2));
    const unsigned alt = (kp.flags & LBM_FLAG_PERIODIC_X) ? off - (unsigned)(dx * kp.nx)
                                                          : other * kp.N;
    const bool out = dx < 0 ? x == 0 : (dx > 0 ? x == kp.nx - 1 : false);
    return out && pn.odd && !turned ? alt : off;
}

// The array from which the offsets of the pair with direction i in row `row`
// count: the array itself, or that row (WIDE).
template <bool WIDE, typename S>
__device__ __forceinline__ S* pair_base(const KParams& kp, S* a, int row) {
    return WIDE ? a + (size_t)row * kp.N : a;
}

// Loads the two nodes' elements of a side, at offsets from `base` (in array a).
template <typename S, bool EDGE>
__device__ __forceinline__ float2 pair_ld(const KParams& kp, const S* __restrict__ a, size_t extent,
                                          const S* base, const PairNodes& pn, unsigned off,
                                          int other, int dx, int dz) {
    float2 v = make_float2(0.0f, 0.0f);
    if constexpr (!EDGE) {
        const unsigned e = pn.n + off;
        if (LBM_IN(kp, LBM_SITE_PAIR_LOAD, a, base + e, 1, extent)) v.x = Store<S>::ld(base + e);
        if (LBM_IN(kp, LBM_SITE_PAIR_LOAD, a, base + e + 32, 1, extent)) v.y = Store<S>::ld(base + e + 32);
    } else {
        // lanes beyond the row read what the last node reads, and drop it: the
        // loads stay unconditional, so none waits for the one before
        const unsigned e0 = pn.clamped(kp, 0) + pair_edge(kp, pn, min(pn.x, kp.nx - 1), off, other, dx, dz);
        const unsigned e1 = pn.clamped(kp, 32) + pair_edge(kp, pn, min(pn.x + 32, kp.nx - 1), off, other, dx, dz);
        if (LBM_IN(kp, LBM_SITE_PAIR_LOAD, a, base + e0, 1, extent)) v.x = Store<S>::ld(base + e0);
        if (LBM_IN(kp, LBM_SITE_PAIR_LOAD, a, base + e1, 1, extent)) v.y = Store<S>::ld(base + e1);
    }
    return v;
}

template <typename S, bool EDGE>
__device__ __forceinline__ void pair_st(const KParams& kp, S* __restrict__ a, size_t extent, S* base,
                                        const PairNodes& pn, unsigned off, int other, int dx,
                                        int dz, float2 v) {
    if constexpr (!EDGE) {
        const unsigned e = pn.n + off;
        if (LBM_IN(kp, LBM_SITE_PAIR_STORE, a, base + e, 1, extent)) Store<S>::st(base + e, v.x);
        if (LBM_IN(kp, LBM_SITE_PAIR_STORE, a, base + e + 32, 1, extent)) Store<S>::st(base + e + 32, v.y);
    } else {
        const unsigned e0 = pn.n + pair_edge(kp, pn, pn.x, off, other, dx, dz);
        const unsigned e1 = pn.n + 32 + pair_edge(kp, pn, pn.x + 32, off, other, dx, dz);
        if (pn.x < kp.nx && LBM_IN(kp, LBM_SITE_PAIR_STORE, a, base + e0, 1, extent))
            Store<S>::st(base + e0, v.x);
        if (pn.x + 32 < kp.nx && LBM_IN(kp, LBM_SITE_PAIR_STORE, a, base + e1, 1, extent))
            Store<S>::st(base + e1, v.y);
    }
}

// Gather of M opposite pairs (rows direction - D0 of an array of ROWS rows):
// f_i from side M, f_(i+1) from side P; the rest population is the caller's.
template <int M, int D0, int ROWS, typename S, bool EDGE, bool WIDE>
__device__ __forceinline__ void pair_gather(const KParams& kp, const S* __restrict__ a,
                                            const PairNodes& pn, const unsigned* off,
                                            float2 (&v)[ROWS]) {
    const size_t ext = (size_t)ROWS * kp.N;
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const int i = 2 * m + 1, cx = cx27(i), cz = cz27(i), row = WIDE ? 0 : i - D0;
        const S* b = pair_base<WIDE>(kp, a, i - D0);
        v[i - D0] = pair_ld<S, EDGE>(kp, a, ext, b, pn, off[2 * m + 1], row, -cx, -cz);
        v[i + 1 - D0] = pair_ld<S, EDGE>(kp, a, ext, b, pn, off[2 * m], row + 1, cx, cz);
    }
}

// Scatter of the post-collision populations: f*_i to side P, f*_(i+1) to side M.
template <int M, int D0, int ROWS, typename S, bool EDGE, bool WIDE>
__device__ __forceinline__ void pair_scatter(const KParams& kp, S* __restrict__ a,
                                             const PairNodes& pn, const unsigned* off,
                                             const float2 (&v)[ROWS]) {
    const size_t ext = (size_t)ROWS * kp.N;
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const int i = 2 * m + 1, cx = cx27(i), cz = cz27(i), row = WIDE ? 0 : i - D0;
        S* b = pair_base<WIDE>(kp, a, i - D0);
        pair_st<S, EDGE>(kp, a, ext, b, pn, off[2 * m], row + 1, cx, cz, v[i - D0]);
        pair_st<S, EDGE>(kp, a, ext, b, pn, off[2 * m + 1], row, -cx, -cz, v[i + 1 - D0]);
    }
}

// The rest population (row 0, direction 0; `a` of any element type).
template <typename T, bool EDGE>
__device__ __forceinline__ float2 pair_ld_rest(const KParams& kp, const T* __restrict__ a,
                                               size_t extent, const PairNodes& pn) {
    return pair_ld<T, EDGE>(kp, a, extent, a, pn, 0u, 0, 0, 0);
}
template <typename T, bool EDGE>
__device__ __forceinline__ void pair_st_rest(const KParams& kp, T* __restrict__ a, size_t extent,
                                             const PairNodes& pn, float2 v) {
    pair_st<T, EDGE>(kp, a, extent, a, pn, 0u, 0, 0, 0, v);
}

}  // namespace lbmgpu
