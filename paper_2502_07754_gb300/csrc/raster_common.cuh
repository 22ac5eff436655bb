// Shared pieces of the rasterisation kernels: double-float projection of a fan
// centre (value path), the shared-memory stage of a chunk of fans' decisions, and the per-pixel
// coverage walk over a staged fan's K triangles with the binary32 decision formulas on
// fan-relative vertex positions.
#pragma once

#include "fan_geom.cuh"
#include "ms_internal.h"

namespace ms {

// Pixels are resolved in descending order of their fragment counts, clamped here.
constexpr int kCountBuckets = 256;
__device__ __forceinline__ int count_bucket(uint32_t n) {
    return n < (uint32_t)kCountBuckets ? (int)n : kCountBuckets - 1;
}

// A pair's pixel rectangle clipped to its tile, relative to the tile's corner: x0 | y0 << 6 |
// (w - 1) << 12 | (h - 1) << 18, bit 31 set; 0 for a pair with no pixel to test.
__device__ __forceinline__ uint32_t pair_geo(int rx0, int ry0, int w, int h) {
    return 0x80000000u | (uint32_t)rx0 | (uint32_t)ry0 << 6 | (uint32_t)(w - 1) << 12 | (uint32_t)(h - 1) << 18;
}

struct SceneDev {
    int W, H;
    const float4 *dec;   // this view's decided vertices (xr, yr, Z or -1, origin), written by binning
    const uint32_t *face_mask;   // per fan, bit j = face j drawn; NULL = all
};

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
// Shared-memory stage (structure of arrays over CH slots)
// ------------------------------------------------------------------------------------

struct Stage {
    int4 *rect;                   // [CH] i0, i1, j0, j1
    uint32_t *flags;              // [CH] bits 0..15 valid triangle, 16..31 negative orientation
    uint32_t *stie, *rtie;        // [CH] top-left tie bits of the spoke / rim directions
    float *ox, *oy;               // [CH] integer origin of the fan's relative positions
    float *vx, *vy;               // [KV][CH] decided vertices relative to the origin
    float2 *sd;                   // [K][CH] spoke directions b_i - c
    float *rdx, *rdy;             // [K][CH] rim directions, lower index to higher
    float *area;                  // [K][CH] |area2|
};

__host__ __device__ __forceinline__ size_t stage_bytes(int CH, int K) {
    return (size_t)CH * (16 + 12 + 8 + 4 * (2 * (K + 1) + 5 * K));
}

__device__ __forceinline__ Stage stage_ptrs(char *base, int CH, int K) {
    const int KV = K + 1;
    Stage s;
    s.rect = reinterpret_cast<int4 *>(base);
    s.flags = reinterpret_cast<uint32_t *>(s.rect + CH);
    s.stie = s.flags + CH;
    s.rtie = s.stie + CH;
    float *f = reinterpret_cast<float *>(s.rtie + CH);
    s.ox = f; f += CH;
    s.oy = f; f += CH;
    s.vx = f; f += KV * CH;
    s.vy = f; f += KV * CH;
    s.sd = reinterpret_cast<float2 *>(f); f += 2 * K * CH;   // (CH is even: 8-byte aligned)
    s.rdx = f; f += K * CH;
    s.rdy = f; f += K * CH;
    s.area = f;
    return s;
}

// OR / min / max over the LPF lanes of a fan's group (lanes lane & ~(LPF-1) .. + LPF-1).
template <int LPF>
__device__ __forceinline__ uint32_t group_or(uint32_t x) {
#pragma unroll
    for (int o = LPF / 2; o > 0; o >>= 1) x |= __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
template <int LPF>
__device__ __forceinline__ float group_min(float x) {
#pragma unroll
    for (int o = LPF / 2; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
template <int LPF>
__device__ __forceinline__ float group_max(float x) {
#pragma unroll
    for (int o = LPF / 2; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// The decision part of stage_fans: decided vertices, spoke and rim directions, areas,
// tie bits, valid-triangle flags and the pixel rectangle of every slot.
template <int LPF>
__device__ __forceinline__ void stage_decisions(const SceneDev &a, const Stage &s, int K, int slot, int sub,
                                                bool active, uint32_t fan) {
    constexpr int CH = 32 / LPF;
    const int KV = K + 1;
    const float4 *dv = a.dec + (size_t)fan * KV;

    uint32_t vmask = 0;
    if (active)
        for (int k = sub; k < KV; k += LPF) {
            const float4 d = __ldg(dv + k);   // the binning pass's decide_vertex, bit for bit
            s.vx[k * CH + slot] = d.x;
            s.vy[k * CH + slot] = d.y;
            if (d.z > 0.0f) vmask |= 1u << k;   // binning marks invalid vertices with Z = -1
            if (k == 0) s.ox[slot] = d.w;
            if (k == 1) s.oy[slot] = d.w;
        }
    vmask = group_or<LPF>(vmask);
    __syncwarp();   // the group's vertex rows are complete
    uint32_t tmask = tri_valid_mask(vmask, K);
    if (a.face_mask && active) tmask &= __ldg(a.face_mask + fan);   // the same word in every lane of the fan
    float mnx = 3.0e38f, mxx = -3.0e38f, mny = 3.0e38f, mxy = -3.0e38f;
    uint32_t flags = 0, stie = 0, rtie = 0;
    if (active) {
        for (int k = sub; k < KV; k += LPF) {
            if (!vertex_used(tmask, k, K)) continue;
            const float x = s.vx[k * CH + slot], y = s.vy[k * CH + slot];
            mnx = fminf(mnx, x); mxx = fmaxf(mxx, x);
            mny = fminf(mny, y); mxy = fmaxf(mxy, y);
        }
        const float xc = s.vx[slot], yc = s.vy[slot];
        for (int j = sub; j < K; j += LPF) {
            const int b = 1 + j, c = 1 + (j + 1 == K ? 0 : j + 1);
            const float xb = s.vx[b * CH + slot], yb = s.vy[b * CH + slot];
            const float xn = s.vx[c * CH + slot], yn = s.vy[c * CH + slot];
            const float sx = __fsub_rn(xb, xc), sy = __fsub_rn(yb, yc);
            float rx, ry;
            if (j + 1 == K) {   // rim (b_{K-1}, b_0): the lower index is b_0
                rx = __fsub_rn(xb, xn);
                ry = __fsub_rn(yb, yn);
            } else {
                rx = __fsub_rn(xn, xb);
                ry = __fsub_rn(yn, yb);
            }
            s.sd[j * CH + slot] = make_float2(sx, sy);
            s.rdx[j * CH + slot] = rx;
            s.rdy[j * CH + slot] = ry;
            const float ar = dec_area2(xc, yc, xb, yb, xn, yn);
            s.area[j * CH + slot] = fabsf(ar);
            if (((tmask >> j) & 1u) && ar != 0.0f) flags |= 1u << j;
            if (ar < 0.0f) flags |= 1u << (16 + j);
            // tie acceptance (E == 0) of each direction and of its reverse
            if (sy < 0.0f || (sy == 0.0f && sx > 0.0f)) stie |= 1u << j;
            if (sy > 0.0f || (sy == 0.0f && sx < 0.0f)) stie |= 1u << (16 + j);
            if (ry < 0.0f || (ry == 0.0f && rx > 0.0f)) rtie |= 1u << j;
            if (ry > 0.0f || (ry == 0.0f && rx < 0.0f)) rtie |= 1u << (16 + j);
        }
    }
    mnx = group_min<LPF>(mnx);
    mxx = group_max<LPF>(mxx);
    mny = group_min<LPF>(mny);
    mxy = group_max<LPF>(mxy);
    flags = group_or<LPF>(flags);
    stie = group_or<LPF>(stie);
    rtie = group_or<LPF>(rtie);
    if (active && sub == 0) {
        const FanRect r = rect_from_bounds_rel(mnx, mxx, mny, mxy, (int)s.ox[slot], (int)s.oy[slot], a.W, a.H);
        s.stie[slot] = stie;
        s.rtie[slot] = rtie;
        s.flags[slot] = (tmask == 0 || r.empty) ? 0u : flags;
        s.rect[slot] = make_int4(r.i0, r.i1, r.j0, r.j1);
    }
}
// Stages CH = 32 / LPF fans into slots 0..CH-1 with the whole warp: the LPF lanes of slot
// lane / LPF share the fan's vertices and triangles (every lane of the warp
// calls this; a lane whose slot is not active does no loads or stores but takes part in
// the shuffles).  The staged words are the same as one lane per fan would write.
template <int LPF>
__device__ __forceinline__ void stage_fans(const SceneDev &a, const Stage &s, int K, int lane, bool active,
                                           uint32_t fan) {
    stage_decisions<LPF>(a, s, K, lane / LPF, lane % LPF, active, fan);
}
// Coverage of the pixel centre (pxc, pyc) by staged fan f: bit j is set when triangle j
// covers it.  Each spoke value is computed once and turned into two pass bits (as the
// edge c -> b_i and as its reverse), so a triangle's two spoke tests are a bit test; only
// triangles passing both get the rim edge.  The result is the conjunction of the three edge
// tests, as stated.  A spoke's bits are its value's sign bit, shifted into the mask by one
// funnel shift; a value of zero (where the top-left tie bits decide) is noticed as a zero
// minimum of the magnitudes and takes the general form below.  The count pass that runs it is
// bound by issue slots (65-72% of them busy): setting two compared and tie-checked bits per
// spoke took about 400 instructions a test; with the sign bits, one 8-byte load per spoke and
// the fan of a test found from start flags instead of a five-step search, 200k fans at 800x800
// went from 1.284 to 1.220 ms (forward and adjoint), 1k fans at 128x128 from 0.54 to 0.48 ms.
template <int KT>
__device__ __forceinline__ uint32_t cover_mask(const Stage &S, int CH, int K, int f, uint32_t flags, float pxc,
                                               float pyc) {
    const float qx = __fsub_rn(pxc, S.vx[f]), qy = __fsub_rn(pyc, S.vy[f]);
    const uint32_t full = (1u << K) - 1u;
    uint32_t N = 0;
    float least = 3.0e38f;
#pragma unroll(KT > 0 ? KT : 1)
    for (int i = K - 1; i >= 0; --i) {   // (descending, so that spoke i lands in bit i)
        const float2 d = S.sd[i * CH + f];
        const float Si = __fsub_rn(__fmul_rn(d.x, qy), __fmul_rn(d.y, qx));
        N = __funnelshift_l(__float_as_uint(Si), N, 1);
        least = fminf(least, fabsf(Si));
    }
    uint32_t P = ~N & full;
    if (least == 0.0f) {   // a centre on a spoke's line
        const uint32_t stie = S.stie[f];
        P = N = 0;
#pragma unroll 1
        for (int i = 0; i < K; ++i) {
            const float2 d = S.sd[i * CH + f];
            const float Si = __fsub_rn(__fmul_rn(d.x, qy), __fmul_rn(d.y, qx));
            const bool z = Si == 0.0f;
            P |= (uint32_t)(Si > 0.0f || (z && ((stie >> i) & 1u))) << i;
            N |= (uint32_t)(Si < 0.0f || (z && ((stie >> (16 + i)) & 1u))) << i;
        }
    }
    const uint32_t Pn = ((P >> 1) | (P << (K - 1))) & full;   // bit j: spoke j+1
    const uint32_t Nn = ((N >> 1) | (N << (K - 1))) & full;
    const uint32_t negm = flags >> 16;
    uint32_t cand = ((P & Nn & ~negm) | (N & Pn & negm)) & flags & full;
    uint32_t hits = 0;
    const uint32_t rtie = S.rtie[f];
    while (cand) {
        const int j = __ffs(cand) - 1;
        cand &= cand - 1;
        const bool neg = (negm >> j) & 1u;
        const bool wrap = (j + 1 == K);
        const int lo = wrap ? 0 : j;
        const float Rc = dec_edge(S.rdx[j * CH + f], S.rdy[j * CH + f], S.vx[(1 + lo) * CH + f],
                                  S.vy[(1 + lo) * CH + f], pxc, pyc);
        // oriented rim: b_j -> b_{j+1} for positive orientation, reversed otherwise
        const bool flip = wrap != neg;
        const float E0 = flip ? -Rc : Rc;
        if (E0 > 0.0f || (E0 == 0.0f && ((rtie >> (flip ? 16 + j : j)) & 1u))) hits |= 1u << j;
    }
    return hits;
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
