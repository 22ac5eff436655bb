// Shared device helpers of the MeshSplats CUDA library (sm_103a).
//
// The "decision" functions evaluate the coverage formulas stated in
// include/meshsplats.h in IEEE binary32 with the round-to-nearest intrinsics (which the
// compiler never fuses into FMAs), on vertex positions taken from a double-float
// projection; the fragment order uses a double-float depth.  The value functions
// (barycentrics, interpolation, compositing, gradients) are free FP32 arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/meshsplats.h"
#include "dfloat.cuh"

namespace ms {

__host__ __device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }

constexpr float kGuardPx = 131072.0f;   // |xs|, |ys| <= 2^17
constexpr int kMaxK = 16;
constexpr uint32_t kSpinLimit = 1u << 20;   // polls before a bounded wait gives up

// Device-side outcome block at the start of every render workspace.
struct Status {
    unsigned long long pairs;        // pairs produced by binning
    unsigned long long culled;       // culled triangles
    unsigned long long extra_passes; // rounds of 32 fragments that pixels took beyond their first
    unsigned long long cap;          // pair capacity of the workspace
    unsigned int timeouts;           // bounded waits that expired
    unsigned int sort_ticket[8];     // virtual block ids of each sort pass (sort_u64)
    unsigned int n_tiles;
    unsigned int sort_bits;
    unsigned long long rect_tests;   // forward rasterisation / resolve work counters
    unsigned long long commits;
    unsigned long long frags;        // fragment records the pixels were given
    unsigned long long frag_cap;     // fragment record capacity of the workspace
    unsigned int tscan_ticket;       // virtual block ids of the tile scan
    alignas(16) unsigned int classes[4];         // pixels of more than 32, 17..32, 9..16, 1..8 fragments
    unsigned int n_items;            // raster work items (<= 64 fans of one tile each)
    unsigned long long items_total;  // work items the tile scan counted
};
// The count pass's coverage masks live in at most this many equal regions, each with its own cursor. A
// cursor counts every test of its region, stored or not: 64 bits, as a small image has one region only and
// wrapped words would hand out stored masks again.
constexpr int kMaskRegions = 128;
static_assert(sizeof(Status) <= 256, "status block");

struct CamDev {
    float R[9];
    float C[3];
    float fx, fy, cx, cy, znear;
    int width, height;
};

inline CamDev make_cam(const ms_camera &c) {
    CamDev d;
    for (int i = 0; i < 9; ++i) d.R[i] = c.R_cw[i];
    for (int i = 0; i < 3; ++i) d.C[i] = c.C[i];
    d.fx = c.fx; d.fy = c.fy; d.cx = c.cx; d.cy = c.cy; d.znear = c.znear;
    d.width = c.width; d.height = c.height;
    return d;
}

// Views of one render call.  Tiles and pixels of all views form one index space: view v
// owns global tiles [tile_base, tile_base + tiles) and pixels [pix_base, pix_base + W H).
// The table travels to the kernels as a __grid_constant__ parameter.
constexpr int kMaxViews = MS_MAX_VIEWS;
struct ViewDev {
    CamDev cam;
    uint32_t tile_base, tiles_x;
    unsigned long long pix_base;
    float *out;               // forward output image, H x W x 4
    const float *dL;          // backward: dL / d image
    const float *out_fwd;     // backward: the forward image
};
struct ViewTable {
    int n;
    ViewDev v[kMaxViews];
};

__device__ __forceinline__ int view_of_tile(const ViewTable &t, uint32_t tile) {
    int lo = 0, hi = t.n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (t.v[mid].tile_base <= tile) lo = mid; else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ int view_of_pixel(const ViewTable &t, unsigned long long pix) {
    int lo = 0, hi = t.n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (t.v[mid].pix_base <= pix) lo = mid; else hi = mid;
    }
    return lo;
}

// ---------------------------------------------------------------------------------
// Decisions
// ---------------------------------------------------------------------------------

// Double-float dot product of a binary32 row R with the double-float vector d: exact
// products of the high parts (FMA residuals), their sum by two-sums, and the remaining
// error terms summed in binary32.
__device__ __forceinline__ dfl df_row_dot(const float *R, dfl d0, dfl d1, dfl d2) {
    const dfl p0 = df_two_prod(R[0], d0.h), p1 = df_two_prod(R[1], d1.h), p2 = df_two_prod(R[2], d2.h);
    const dfl s = df_two_sum(p0.h, p1.h);
    const dfl t = df_two_sum(s.h, p2.h);
    const float l = __fadd_rn(__fadd_rn(__fadd_rn(s.l, t.l), __fadd_rn(__fadd_rn(p0.l, p1.l), p2.l)),
                              fmaf(R[0], d0.l, fmaf(R[1], d1.l, __fmul_rn(R[2], d2.l))));
    return df_fast_two_sum(t.h, l);
}

// f (N / Z) + c in double-float, the quotient from one reciprocal of Z.h and a
// double-float residual correction.
__device__ __forceinline__ dfl df_screen_coord(dfl N, dfl Z, float rz, float f, float c) {
    const float q1 = __fmul_rn(N.h, rz);
    const float r = __fadd_rn(fmaf(-q1, Z.h, N.h), fmaf(-q1, Z.l, N.l));
    const dfl q = df_fast_two_sum(q1, __fmul_rn(r, rz));
    dfl a = df_mul_f(q, f);
    return df_add_f(a, c);
}

// Camera-space position (X, Y, Z) and screen position (x, y) of a world point, all in
// double-float: d = p - C is exact, then the rotation and the pinhole division.
struct DfVert {
    dfl X, Y, Z, x, y;
};
__device__ __forceinline__ DfVert df_project(const CamDev &c, float px, float py, float pz) {
    const dfl d0 = df_two_sum(px, -c.C[0]), d1 = df_two_sum(py, -c.C[1]), d2 = df_two_sum(pz, -c.C[2]);
    DfVert o;
    o.X = df_row_dot(c.R, d0, d1, d2);
    o.Y = df_row_dot(c.R + 3, d0, d1, d2);
    o.Z = df_row_dot(c.R + 6, d0, d1, d2);
    const float rz = __frcp_rn(o.Z.h);
    o.x = df_screen_coord(o.X, o.Z, rz, c.fx, c.cx);
    o.y = df_screen_coord(o.Y, o.Z, rz, c.fy, c.cy);
    return o;
}

// A vertex as the coverage decisions see it: the double-float screen position rounded to
// binary32 (xs, ys) and relative to its fan's integer origin (xr, yr) = nearest binary32
// value of (x - ox, y - oy), its rounded depth Z, and the validity rule on the rounded
// values (Z > znear, |xs|, |ys| <= 2^17).
struct DVert {
    float xs, ys, xr, yr, Z;
    bool valid;
};

// Nearest binary32 value of v - o for an integer-valued binary32 o (exact two-sum of the
// high part, then the low parts).
__device__ __forceinline__ float df_offset(dfl v, float o) {
    const dfl s = df_two_sum(v.h, -o);
    return __fadd_rn(s.h, __fadd_rn(s.l, v.l));
}

__device__ __forceinline__ DVert decide_vertex(const CamDev &c, const DfVert &v, float ox, float oy) {
    DVert o;
    o.xs = df_round(v.x);
    o.ys = df_round(v.y);
    o.xr = df_offset(v.x, ox);
    o.yr = df_offset(v.y, oy);
    o.Z = df_round(v.Z);
    o.valid = (o.Z > c.znear) && (fabsf(o.xs) <= kGuardPx) && (fabsf(o.ys) <= kGuardPx);
    return o;
}

__device__ __forceinline__ float dec_area2(float xa, float ya, float xb, float yb, float xc, float yc) {
    return __fsub_rn(__fmul_rn(__fsub_rn(xb, xa), __fsub_rn(yc, ya)),
                     __fmul_rn(__fsub_rn(yb, ya), __fsub_rn(xc, xa)));
}

// Canonical edge value from vertex lo (lower index) to hi, with the direction
// (ex, ey) = (hi - lo) precomputed.
__device__ __forceinline__ float dec_edge(float ex, float ey, float lx, float ly, float px, float py) {
    return __fsub_rn(__fmul_rn(ex, __fsub_rn(py, ly)), __fmul_rn(ey, __fsub_rn(px, lx)));
}

// ---------------------------------------------------------------------------------
// 32-byte records: one 256-bit access of sm_100-class GPUs, p 32-byte aligned.  Used where a pass waits
// on its records (resolve and its adjoint: view of 200k fans 878 -> 862 us; splat fill); the fan fill's and
// the chain's accesses gain nothing by it.
// ---------------------------------------------------------------------------------

__device__ __forceinline__ void ld_rec(const float4 *p, float4 &a, float4 &b) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                 : "l"(p));
}
__device__ __forceinline__ void st_rec(float4 *p, const float4 a, const float4 b) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w),
                 "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// ---------------------------------------------------------------------------------
// Bounded waits
// ---------------------------------------------------------------------------------

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_u64(unsigned long long *p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_u32(uint32_t *p, uint32_t v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

}  // namespace ms
