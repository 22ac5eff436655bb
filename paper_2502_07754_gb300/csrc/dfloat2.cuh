// Double-float arithmetic on pairs of values: the packed f32x2 instructions of sm_100-class GPUs
// round each half like the scalar instruction, so every function here gives the bits of its scalar
// form (dfloat.cuh, ms_common.cuh) for both values in half the instructions.  A difference is an
// FMA by -1; where a negated term is what the FMA needs, the sum is carried negated (rounding is
// symmetric).
#pragma once

#include "ms_common.cuh"

namespace ms {

struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2_pack(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_get(F2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) { return f2_fma(b, f2_pack(-1.0f, -1.0f), a); }
__device__ __forceinline__ F2 f2_neg(F2 a) { return f2_mul(a, f2_pack(-1.0f, -1.0f)); }

struct dfl2 {
    F2 h, l;
};
__device__ __forceinline__ dfl2 df2_two_sum(F2 a, F2 b) {
    const F2 s = f2_add(a, b), bb = f2_sub(s, a);
    return dfl2{s, f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb))};
}
__device__ __forceinline__ dfl2 df2_fast_two_sum(F2 a, F2 b) {
    const F2 s = f2_add(a, b);
    return dfl2{s, f2_sub(b, f2_sub(s, a))};
}

// df_row_dot (nd: the negated high parts of d).
__device__ __forceinline__ dfl2 df2_row_dot(F2 R0, F2 R1, F2 R2, const dfl2 d[3], const F2 nd[3]) {
    const F2 p0 = f2_mul(R0, d[0].h), p1 = f2_mul(R1, d[1].h), p2 = f2_mul(R2, d[2].h);
    const F2 n0 = f2_fma(R0, nd[0], p0), n1 = f2_fma(R1, nd[1], p1), n2 = f2_fma(R2, nd[2], p2);   // -residuals
    const dfl2 s = df2_two_sum(p0, p1), t = df2_two_sum(s.h, p2);
    const F2 l = f2_add(f2_sub(f2_add(s.l, t.l), f2_add(f2_add(n0, n1), n2)),
                        f2_fma(R0, d[0].l, f2_fma(R1, d[1].l, f2_mul(R2, d[2].l))));
    return df2_fast_two_sum(t.h, l);
}

// df_screen_coord (rz, nrz: the reciprocals of Z.h and their negatives).
__device__ __forceinline__ dfl2 df2_screen_coord(dfl2 N, dfl2 Z, F2 rz, F2 nrz, F2 f, F2 c) {
    const F2 q1 = f2_mul(N.h, rz), nq1 = f2_mul(N.h, nrz);
    const F2 r = f2_add(f2_fma(nq1, Z.h, N.h), f2_fma(nq1, Z.l, N.l));
    const F2 t = f2_mul(r, rz);
    const F2 qh = f2_add(q1, t), nqh = f2_sub(nq1, t), nql = f2_sub(f2_sub(qh, q1), t);
    const F2 p = f2_mul(qh, f), npl = f2_fma(nql, f, f2_fma(nqh, f, p));   // the product and its negated low part
    const F2 ah = f2_sub(p, npl), nal = f2_add(npl, f2_sub(ah, p));
    const dfl2 s = df2_two_sum(ah, c);
    return df2_fast_two_sum(s.h, f2_sub(s.l, nal));
}

// A camera's constants, each in both halves.
struct Cam2 {
    F2 nC[3], R[9], fx, fy, cx, cy;
};
__device__ __forceinline__ Cam2 cam2(const CamDev &c) {
    Cam2 o;
#pragma unroll
    for (int i = 0; i < 3; ++i) o.nC[i] = f2_pack(-c.C[i], -c.C[i]);
#pragma unroll
    for (int i = 0; i < 9; ++i) o.R[i] = f2_pack(c.R[i], c.R[i]);
    o.fx = f2_pack(c.fx, c.fx);
    o.fy = f2_pack(c.fy, c.fy);
    o.cx = f2_pack(c.cx, c.cx);
    o.cy = f2_pack(c.cy, c.cy);
    return o;
}

// decide_vertex(df_project) of the points p and q.
__device__ __forceinline__ void decide_vertex2(const CamDev &cam, const Cam2 &c, const float *p, const float *q, F2 nox,
                                               F2 noy, DVert &a, DVert &b) {
    dfl2 d[3];
    F2 nd[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        d[r] = df2_two_sum(f2_pack(p[r], q[r]), c.nC[r]);
        nd[r] = f2_neg(d[r].h);
    }
    const dfl2 X = df2_row_dot(c.R[0], c.R[1], c.R[2], d, nd), Y = df2_row_dot(c.R[3], c.R[4], c.R[5], d, nd);
    const dfl2 Z = df2_row_dot(c.R[6], c.R[7], c.R[8], d, nd);
    const float2 zh = f2_get(Z.h);
    const F2 rz = f2_pack(__frcp_rn(zh.x), __frcp_rn(zh.y)), nrz = f2_neg(rz);
    const dfl2 x = df2_screen_coord(X, Z, rz, nrz, c.fx, c.cx), y = df2_screen_coord(Y, Z, rz, nrz, c.fy, c.cy);
    const dfl2 sx = df2_two_sum(x.h, nox), sy = df2_two_sum(y.h, noy);
    const float2 xs = f2_get(f2_add(x.h, x.l)), ys = f2_get(f2_add(y.h, y.l)), z = f2_get(f2_add(Z.h, Z.l));
    const float2 xr = f2_get(f2_add(sx.h, f2_add(sx.l, x.l))), yr = f2_get(f2_add(sy.h, f2_add(sy.l, y.l)));
    a = DVert{xs.x, ys.x, xr.x, yr.x, z.x, z.x > cam.znear && fabsf(xs.x) <= kGuardPx && fabsf(ys.x) <= kGuardPx};
    b = DVert{xs.y, ys.y, xr.y, yr.y, z.y, z.y > cam.znear && fabsf(xs.y) <= kGuardPx && fabsf(ys.y) <= kGuardPx};
}

}  // namespace ms
