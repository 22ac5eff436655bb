// Shared pieces of the rasterisation kernels: a pair's rectangle word, the double-float projection
// of a fan centre (value path), and the FP64 formulas of the source Gaussians.
#pragma once

#include "fan_geom.cuh"
#include "ms_internal.h"

namespace ms {

// Pixels are resolved in descending order of their fragment counts, clamped here.
constexpr int kCountBuckets = 256;
__device__ __forceinline__ int count_bucket(uint32_t n) {
    return n < (uint32_t)kCountBuckets ? (int)n : kCountBuckets - 1;
}

// The passes over the work items launch a warp an item up to kItemBlocks blocks; beyond, kStrideBlocks
// blocks stride over the items.  The items are counted on the device, their capacity is many times what a
// scene needs, and a block without an item still takes a launch slot: the 16 views of 3M fans have 0.9M items
// and room for 6.3M, and forward and adjoint took 19.7 ms with a warp for each, 17.5 ms with the stride.
// Below the bound the loop costs more (2% of 8 views of 250k Gaussians) than the empty blocks do.
constexpr int64_t kItemBlocks = 256 * 1024, kStrideBlocks = 64 * 1024;

// A pair's pixel rectangle clipped to its tile, relative to the tile's corner: x0 | y0 << 6 |
// (w - 1) << 12 | (h - 1) << 18, bit 31 set; 0 for a pair with no pixel to test.
__device__ __forceinline__ uint32_t pair_geo(int rx0, int ry0, int w, int h) {
    return 0x80000000u | (uint32_t)rx0 | (uint32_t)ry0 << 6 | (uint32_t)(w - 1) << 12 | (uint32_t)(h - 1) << 18;
}

// ------------------------------------------------------------------------------------
// Double-float helpers of the value path (Knuth two-sum, FMA two-product)
// ------------------------------------------------------------------------------------

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e) {
    p = __fmul_rn(a, b);
    e = fmaf(a, b, -p);
}
// Row of R_cw applied to (d_hi + d_lo), as hi + lo.
__device__ __forceinline__ void df_dot(const float *R, const float dh[3], const float dl[3], float &h, float &l) {
    float p0, q0, p1, q1, p2, q2, s, e1, e2;
    two_prod(R[0], dh[0], p0, q0);
    two_prod(R[1], dh[1], p1, q1);
    two_prod(R[2], dh[2], p2, q2);
    two_sum(p0, p1, s, e1);
    two_sum(s, p2, h, e2);
    l = ((e1 + e2) + (q0 + q1 + q2)) + (R[0] * dl[0] + R[1] * dl[1] + R[2] * dl[2]);
}
// f * (X / Z) + c as hi + lo, with X, Z given as hi + lo.
__device__ __forceinline__ void df_screen(float Xh, float Xl, float Zh, float Zl, float f, float c, float &h,
                                          float &l) {
    const float q1 = Xh / Zh;
    const float r = fmaf(-q1, Zh, Xh) + (Xl - q1 * Zl);
    const float q2 = r / Zh;
    float a1, a2, e;
    two_prod(f, q1, a1, a2);
    a2 = fmaf(f, q2, a2);
    two_sum(a1, c, h, e);
    l = e + a2;
}

// View-space centre of a fan (hi parts) and its double-float screen position.  The
// other vertices are placed by their exact world offsets from the centre, so screen
// positions relative to a pixel carry ~1e-6 px error instead of the ~1e-4 px of a
// plain binary32 projection at 1080p.
struct CentreProj {
    float Xh, Yh, Zh, Xl, Yl, Zl;
    float xh, xl, yh, yl;
};
__device__ __forceinline__ CentreProj project_centre(const CamDev &c, const float m[3]) {
    float dh[3], dl[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) two_sum(m[r], -c.C[r], dh[r], dl[r]);
    CentreProj o;
    df_dot(c.R, dh, dl, o.Xh, o.Xl);
    df_dot(c.R + 3, dh, dl, o.Yh, o.Yl);
    df_dot(c.R + 6, dh, dl, o.Zh, o.Zl);
    df_screen(o.Xh, o.Xl, o.Zh, o.Zl, c.fx, c.cx, o.xh, o.xl);
    df_screen(o.Yh, o.Yl, o.Zh, o.Zl, c.fy, c.cy, o.yh, o.yl);
    return o;
}
__device__ __forceinline__ void vertex_offset(const CamDev &c, const CentreProj &cp, const float d[3], float &du,
                                              float &dv, float &X, float &Y, float &Z) {
    const float dX = c.R[0] * d[0] + c.R[1] * d[1] + c.R[2] * d[2];
    const float dY = c.R[3] * d[0] + c.R[4] * d[1] + c.R[5] * d[2];
    const float dZ = c.R[6] * d[0] + c.R[7] * d[1] + c.R[8] * d[2];
    X = cp.Xh + dX;
    Y = cp.Yh + dY;
    Z = cp.Zh + dZ;
    const float den = 1.0f / (Z * cp.Zh);
    du = c.fx * (dX * cp.Zh - cp.Xh * dZ) * den;
    dv = c.fy * (dY * cp.Zh - cp.Yh * dZ) * den;
}

// Camera-space offset R (p - m) of a vertex from its fan centre, in double-float (the
// world difference of two binary32 values is exact as a two-sum).
struct DfVec {
    dfl x, y, z;
};
__device__ __forceinline__ DfVec df_view_offset(const CamDev &c, const float m[3], const float *p) {
    const dfl d0 = df_two_sum(__ldg(p), -m[0]), d1 = df_two_sum(__ldg(p + 1), -m[1]);
    const dfl d2 = df_two_sum(__ldg(p + 2), -m[2]);
    return DfVec{df_row_dot(c.R, d0, d1, d2), df_row_dot(c.R + 3, d0, d1, d2), df_row_dot(c.R + 6, d0, d1, d2)};
}

// ------------------------------------------------------------------------------------
// Source-Gaussian splats in FP64 (the splat image is the reference that the fans approximate;
// splat_raster.cu takes these formulas where its faster forms leave a case open)
// ------------------------------------------------------------------------------------

// The flat Gaussian g: rotation from the normalised quaternion (w, x, y, z), the two kept
// axes by the same rule as the fan conversion.
struct SplatAxes {
    double m[3], ra[3], rb[3], sa, sb;   // centre, kept unit axes (world), their scales
    float sigma;
};
__device__ __forceinline__ SplatAxes splat_axes(const SplatSrc &src, int64_t g) {
    SplatAxes o;
    const float4 qf = *reinterpret_cast<const float4 *>(src.quats + 4 * (size_t)g);
    const double qn = sqrt((double)qf.x * qf.x + (double)qf.y * qf.y + (double)qf.z * qf.z + (double)qf.w * qf.w);
    const double w = qf.x / qn, x = qf.y / qn, y = qf.z / qn, z = qf.w / qn;
    const double R[9] = {1 - 2 * (y * y + z * z), 2 * (x * y - w * z),     2 * (x * z + w * y),
                         2 * (x * y + w * z),     1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                         2 * (x * z - w * y),     2 * (y * z + w * x),     1 - 2 * (x * x + y * y)};
    const float *ls = src.log_scales + 3 * (size_t)g;
    const float s0 = ls[0], s1 = ls[1], s2 = ls[2];
    int drop = 0;
    if (src.axis_rule == 1) {
        float sm = s0;
        if (s1 < sm) { drop = 1; sm = s1; }
        if (s2 < sm) drop = 2;
    }
    const int ia = drop == 0 ? 1 : 0, ib = drop == 2 ? 1 : 2;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        o.m[r] = (double)src.means[3 * (size_t)g + r];
        o.ra[r] = ia == 0 ? R[3 * r] : R[3 * r + 1];
        o.rb[r] = ib == 2 ? R[3 * r + 2] : R[3 * r + 1];
    }
    o.sa = exp((double)(ia == 0 ? s0 : s1));
    o.sb = exp((double)(ib == 2 ? s2 : s1));
    o.sigma = src.opacity[g];
    return o;
}

struct SplatSlot {
    double mc[3], ua[3], ub[3], n[3];   // camera-space centre, kept unit axes, plane normal
    double mcn, sa, sb;                 // mc . n, the two kept scales
    float sigma;
};
// The Gaussian in the camera frame of c.
__device__ __forceinline__ SplatSlot splat_in_view(const SplatAxes &ax, const CamDev &c) {
    SplatSlot o;
    const double dm[3] = {ax.m[0] - (double)c.C[0], ax.m[1] - (double)c.C[1], ax.m[2] - (double)c.C[2]};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const double R0 = c.R[3 * r], R1 = c.R[3 * r + 1], R2 = c.R[3 * r + 2];
        o.mc[r] = R0 * dm[0] + R1 * dm[1] + R2 * dm[2];
        o.ua[r] = R0 * ax.ra[0] + R1 * ax.ra[1] + R2 * ax.ra[2];
        o.ub[r] = R0 * ax.rb[0] + R1 * ax.rb[1] + R2 * ax.rb[2];
    }
    o.n[0] = o.ua[1] * o.ub[2] - o.ua[2] * o.ub[1];
    o.n[1] = o.ua[2] * o.ub[0] - o.ua[0] * o.ub[2];
    o.n[2] = o.ua[0] * o.ub[1] - o.ua[1] * o.ub[0];
    o.mcn = o.mc[0] * o.n[0] + o.mc[1] * o.n[1] + o.mc[2] * o.n[2];
    o.sa = ax.sa;
    o.sb = ax.sb;
    o.sigma = ax.sigma;
    return o;
}

// Ray of pixel centre (px, py) against splat s: kept when the hit lies in front of the
// near plane and inside the truncation ellipse; t = view depth of the hit (rounded to
// binary32 as the order key), a = sigma exp(-(u^2/sa^2 + v^2/sb^2)/2).
__device__ __forceinline__ bool splat_hit(const SplatSlot &s, const CamDev &c, double trunc, double px, double py,
                                          float &t, float &a) {
    const double d0 = (px - (double)c.cx) / (double)c.fx, d1 = (py - (double)c.cy) / (double)c.fy;
    const double den = d0 * s.n[0] + d1 * s.n[1] + s.n[2];
    if (den == 0.0) return false;
    const double tt = s.mcn / den;
    if (!(tt > (double)c.znear)) return false;
    const double w0 = tt * d0 - s.mc[0], w1 = tt * d1 - s.mc[1], w2 = tt - s.mc[2];
    const double u = w0 * s.ua[0] + w1 * s.ua[1] + w2 * s.ua[2];
    const double v = w0 * s.ub[0] + w1 * s.ub[1] + w2 * s.ub[2];
    const double ru = u / (trunc * s.sa), rv = v / (trunc * s.sb);
    if (!(ru * ru + rv * rv <= 1.0)) return false;
    t = (float)tt;
    a = (float)((double)s.sigma * exp(-0.5 * (u * u / (s.sa * s.sa) + v * v / (s.sb * s.sb))));
    return true;
}

}  // namespace ms
