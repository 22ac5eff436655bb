// Per-fan screen-space setup shared by binning and the composite kernels, so that
// both derive bit-identical pixel rectangles and depth keys for a fan.
#pragma once

#include "ms_common.cuh"

namespace ms {

struct FanRect {
    int i0, i1, j0, j1;   // inclusive pixel range that may hold covered pixel centres
    bool empty;
};

// Margin around the vertices' bounds within which a centre may still be accepted.  Bound on
// the binary32 edge test: a centre p it accepts lies within 2.1 * 2^-24 * (|p - a|_1) of each
// edge line (a = the edge's lower vertex), plus the turn of the rounded edge direction --
// together below 2^-21 of the bounds' width and height, < 0.07 + 0.03 px for anything in the
// +-2^17 guard band -- and the absolute positions that binning takes its bounds from are
// rounded by at most 2^-7 px there.  1/32 px plus 2^-20 of the extent exceeds both; a quarter
// pixel is the most that any fan needs.  (The three lines' strips can meet further out only past
// the tip of a sliver; a centre there is outside the triangle and is left out.  A constant quarter
// pixel around fans of about a pixel doubles the centres tested: 3M fans in 16 views, 160M tests and
// 55.6M pairs with it, 96M and 42.4M with this one; the batch step 32.86 -> 28.81 ms.)
__device__ __forceinline__ float rect_margin(float mnx, float mxx, float mny, float mxy) {
    return fminf(0.25f, 0.03125f + 0x1p-20f * ((mxx - mnx) + (mxy - mny)));
}

// Pixel centres i + 0.5 within [min x - margin, max x + margin] (and the same in y) of the
// vertices of the fan's valid triangles, so no covered centre falls outside.  min/max are
// order independent, so every caller that feeds the same vertex set gets the same rectangle.
__device__ __forceinline__ FanRect rect_from_bounds(float mnx, float mxx, float mny, float mxy, int W, int H) {
    const float g = rect_margin(mnx, mxx, mny, mxy);
    FanRect r;
    r.i0 = max((int)ceilf(mnx - (0.5f + g)), 0);
    r.i1 = min((int)floorf(mxx - (0.5f - g)), W - 1);
    r.j0 = max((int)ceilf(mny - (0.5f + g)), 0);
    r.j1 = min((int)floorf(mxy - (0.5f - g)), H - 1);
    r.empty = r.i0 > r.i1 || r.j0 > r.j1;
    return r;
}

// rect_from_bounds for bounds given relative to the integer origin (ox, oy): identical
// pixel arithmetic in the relative frame, shifted by the origin.
__device__ __forceinline__ FanRect rect_from_bounds_rel(float mnx, float mxx, float mny, float mxy, int ox, int oy,
                                                        int W, int H) {
    const float g = rect_margin(mnx, mxx, mny, mxy);
    FanRect r;
    r.i0 = max((int)ceilf(mnx - (0.5f + g)) + ox, 0);
    r.i1 = min((int)floorf(mxx - (0.5f - g)) + ox, W - 1);
    r.j0 = max((int)ceilf(mny - (0.5f + g)) + oy, 0);
    r.j1 = min((int)floorf(mxy - (0.5f - g)) + oy, H - 1);
    r.empty = r.i0 > r.i1 || r.j0 > r.j1;
    return r;
}

// Triangle j of a fan is valid when the centre and both of its boundary vertices are.
__device__ __forceinline__ uint32_t tri_valid_mask(uint32_t vmask, int K) {
    uint32_t t = 0;
    if (vmask & 1u)
        for (int j = 0; j < K; ++j) {
            const int jn = j + 1 == K ? 0 : j + 1;
            if (((vmask >> (1 + j)) & 1u) && ((vmask >> (1 + jn)) & 1u)) t |= 1u << j;
        }
    return t;
}

// Whether vertex k (0 = centre, 1 + i = boundary i) belongs to a valid triangle.
__device__ __forceinline__ bool vertex_used(uint32_t tmask, int k, int K) {
    if (k == 0) return tmask != 0;
    const int i = k - 1, ip = i == 0 ? K - 1 : i - 1;
    return ((tmask >> i) & 1u) || ((tmask >> ip) & 1u);
}

}  // namespace ms
