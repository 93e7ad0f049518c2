// Neighbour ids from a site's record (see SiteLinks in internal.h).
#pragma once

#include "internal.h"
#include "lattice.cuh"

namespace lbm {

__host__ __device__ __forceinline__ int low16(int x) { return static_cast<short>(x & 0xffff); }
__host__ __device__ __forceinline__ int high16(int x) { return x >> 16; }

// Whether x + xi_Q is a pore site.
template <int Q>
__host__ __device__ __forceinline__ bool link_has(const SiteLinks& l) {
    return (l.a.w >> (Q - 1)) & 1;
}

// Site id of x + xi_Q where that is a pore site (and the record is regular):
// in a row with rank r at its middle voxel, r there, r - 1 at dx = -1, and
// r + 1 at dx = +1, or r if the middle voxel is solid.
template <int Q>
__host__ __device__ __forceinline__ int link_id(int n, const SiteLinks& l) {
    constexpr int x = cx(Q), y = cy(Q), z = cz(Q);
    if constexpr (y == 0 && z == 0) {
        return n + x;
    } else {
        int row;
        if constexpr (z == 0) row = n + (y > 0 ? low16(l.a.x) : high16(l.a.x));
        else if constexpr (y == 0) row = z > 0 ? l.a.y : l.a.z;
        else if constexpr (z > 0) row = l.a.y + (y > 0 ? low16(l.b.x) : high16(l.b.x));
        else row = l.a.z + (y > 0 ? low16(l.b.y) : high16(l.b.y));
        if constexpr (x < 0) return row - 1;
        if constexpr (x > 0) {
            constexpr int mid = z == 0 ? (y > 0 ? 3 : 4) : (z > 0 ? 5 : 6);   // the row's middle voxel
            return row + static_cast<int>(link_has<mid>(l));
        }
        return row;
    }
}

// Where direction Q is written to (and opp(Q) read from) by site n at an odd step: row
// Q at x + xi_Q, with its id, or where there is none row opp(Q) at n itself, as an
// offset from row Q. Opposite rows are neighbours, so the offset fits 32 bits for any
// number of sites below 2^31, without a sign where opp(Q) follows Q, with one where it
// precedes it.
template <int Q>
__host__ __device__ __forceinline__ unsigned slot_word(bool has, int id, int n, int pitch) {
    const unsigned p = static_cast<unsigned>(pitch);
    return has ? static_cast<unsigned>(id) : static_cast<unsigned>(n) + (opp(Q) > Q ? p : 0u - p);
}
template <int Q, class T>
__host__ __device__ __forceinline__ T* slot_at(T* row, unsigned word) {   // row: row Q
    if constexpr (opp(Q) > Q) return row + word;
    else return row + static_cast<int>(word);
}

#ifdef __CUDACC__
// Ids of the six face neighbours of site n into nb[1..6], -1 where there is none.
template <int K>
__device__ __forceinline__ void face_neighbours(const DomainView& d, int n, int (&nb)[K]) {
    const int4 a = __ldg(d.link_a + n);
    if (a.w & kIrregular) {
        const int v = __ldg(d.site_vox + n);
        static_for<1, Q7>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            nb[q] = __ldg(d.vsite + v + stencil_off(d, q));
        });
    } else {
        const SiteLinks l{a, make_int2(0, 0)};
        static_for<1, Q7>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            nb[q] = link_has<q>(l) ? link_id<q>(n, l) : -1;
        });
    }
}
#endif

}  // namespace lbm
