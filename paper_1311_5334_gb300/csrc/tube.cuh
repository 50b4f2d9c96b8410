// tube.cuh -- the cell cover of a seed's tube and the exact membership test.
//
// Membership (Section 2, Fig. 4b; exact): grain k lies on the seed line
// through g_a with direction w = g_b - g_a iff
//     |(g_k - g_a) x w|^2 <= r^2 |w|^2 .
// Cross-product components are exact int32 under the parameter precondition
// (|d_e w_f| + |d_f w_e| < 2^31); each square is below 2^62, so their sum is
// below 3 * 2^62 and exact in unsigned 64 bits, and so is r^2 |w|^2 (the
// parameters keep 3 r^2 seed_max^2 below 2^63).
//
// Cover.  The tube is an infinite cylinder across the view.  A grain p in the
// tube has a foot point q(t) = g_a + t w with |p - q| <= r, so on every axis
// |p_e - q_e(t)| <= r.  Grains are grouped in rows (cy, cz) of cells along x,
// each row a contiguous range of the cell-ordered grain array.  For each row
// the parameter interval where q_y and q_z can serve a grain of that row is
// intersected with the interval where q stays near the view; over it q_x
// spans an interval, widened by r, that gives the row's run of x cells.  All
// bounds are computed in FP32 and widened by r + COVER_PAD: with coordinates
// below 2^22 every rounding error is under one unit while the extra pad is
// COVER_PAD units, so the cover is a superset of the tube and the exact test
// decides.  The cover depends on the cell size; the count does not.
#pragma once
#include "common.cuh"

namespace et {

constexpr float COVER_PAD = 4.0f;

// Grain g against the line of moment m = g_a x w: (g - g_a) x w = g x w - m.
// The components of m are exact int32 like those of the difference; sums on the
// way may wrap, so they are unsigned.  Six multiply-adds, where differences
// from g_a first took three subtractions and six.
__device__ __forceinline__ bool in_tube(int4 g, int3 m, int3 w, long long R) {
    const u32 gx = (u32)g.x, gy = (u32)g.y, gz = (u32)g.z, wx = (u32)w.x, wy = (u32)w.y, wz = (u32)w.z;
    const int cx = (int)(gy * wz - (gz * wy + (u32)m.x));
    const int cy = (int)(gz * wx - (gx * wz + (u32)m.y));
    const int cz = (int)(gx * wy - (gy * wx + (u32)m.z));
    const unsigned long long s = (unsigned long long)((long long)cx * cx) +
                                 (unsigned long long)((long long)cy * cy) +
                                 (unsigned long long)((long long)cz * cz);
    return s <= (unsigned long long)R;
}

__device__ __forceinline__ int floor_i(float x) { return __float2int_rd(x); }

}  // namespace et
