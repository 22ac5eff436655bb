// Rasterisation of the source Gaussians themselves (ms_splat_render) over the tile lists of
// their circumscribing polygons: a count pass and a fill pass like the fans' (raster.cu,
// fill.cu), with the ray / splat test in place of the triangle coverage.
//
// A splat is the flat Gaussian on its plane: the pixel's ray meets the plane at view depth t,
// and is kept when t lies beyond the near plane and the hit inside the truncation ellipse;
// its opacity is sigma exp(-(u^2 / sa^2 + v^2 / sb^2) / 2).  These are stated in FP64
// (splat_hit in raster_common.cuh), whose rate here is a small fraction of binary32's, so:
//  * splat_setup_kernel writes, per view and Gaussian, the test as rational functions of the
//    pixel's offset (dx, dy) from the centre's screen position: with d the ray, n the normal
//    and D = n . d / n . d_centre = 1 + d1 dx + d2 dy,
//      t = Z_c / D,  u / sa = (a1 dx + a2 dy) / D,  v / sb = (b1 dx + b2 dy) / D
//    (u and v vanish at the centre, so no term cancels), every coefficient rounded from FP64
//    to a double-float;
//  * the decision is taken in binary32 where it is certain by a margin of 32 units of 2^-24 of
//    the summed magnitudes, and by the FP64 test itself in the few cases left (a few per
//    100,000, plus every degenerate splat: its coefficients are not finite);
//  * depth and opacity of a hit are computed in double-float by whole warps of hits, with a bound on
//    their error: that of D's summed magnitudes, of the centre's rounded position times the slopes
//    (a centre at 30000 px of a plane 5 px from edge-on is off by 2^-35 of D), and of FP64's own
//    cancellation edge-on. Where it exceeds 2^-40 of D, and where the depth lies that close to a tie of its
//    rounding to the binary32 order key, the FP64 values are taken.  So decisions and order
//    keys are those of the FP64 test, and opacities are within 2^-30 of its values before the last
//    rounding.
// What bounds it: issue slots.  250k Gaussians into eight 1080p views (120M tests, 68M hits): setup
// 0.60 ms (FP64), count 0.88 ms, fill 1.61 ms; with every test, setup and value in FP64 the two
// passes took 20 and 34 ms.
#include "raster_common.cuh"

namespace ms {

namespace {

constexpr int kSplatWarps = 2;

struct SplatArgs {
    ViewTable vt;
    SplatSrc spl;
    int64_t N;
    const uint32_t *list;
    const uint4 *items;
    uint32_t *icnt;
    const uint32_t *offsets;
    uint32_t *counts;
    float4 *frags;
    int64_t frag_cap;
    Status *st;
    const float4 *dec;      // [view][vertex] decided polygon vertices
    int64_t V;
    unsigned long long *tests;   // [kMaskRegions] tests, in parts
    uint2 *pinfo;           // per pair: (0, rectangle within the tile; 0 if no centre is hit)
    const float4 *coef;     // [view][Gaussian][5]
    float r2;               // squared truncation radius in scales
};

__device__ __forceinline__ float2 split(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}

// Coefficients of every (view, Gaussian), one thread a Gaussian: [0] centre x, y; [1] a1, a2;
// [2] b1, b2; [3] d1, d2 (double-float pairs); [4] Z_c, sigma, error of D (and 2^-8 of that of u and v) that
// does not depend on the pixel.
constexpr int kSetupThreads = 128;
__global__ void __launch_bounds__(kSetupThreads) splat_setup_kernel(const SplatSrc s, int64_t N,
                                                                    const __grid_constant__ ViewTable vt,
                                                                    float4 *__restrict__ coef) {
    const int64_t g = (int64_t)blockIdx.x * kSetupThreads + threadIdx.x;
    if (g >= N) return;
    const SplatAxes ax = splat_axes(s, g);
    const double isa = 1.0 / ax.sa, isb = 1.0 / ax.sb;
    for (int v = 0; v < vt.n; ++v) {
        const CamDev &c = vt.v[v].cam;
        const SplatSlot o = splat_in_view(ax, c);
        const double iZ = 1.0 / o.mc[2], fx = c.fx, fy = c.fy;
        const double iD = 1.0 / (o.mcn * iZ);
        const double mua = o.mc[0] * o.ua[0] + o.mc[1] * o.ua[1] + o.mc[2] * o.ua[2];
        const double mub = o.mc[0] * o.ub[0] + o.mc[1] * o.ub[1] + o.mc[2] * o.ub[2];
        const double ix = iD / fx, iy = iD / fy;
        float4 *w = coef + 5 * ((size_t)v * N + g);
        const float2 xc = split(fx * (o.mc[0] * iZ) + c.cx), yc = split(fy * (o.mc[1] * iZ) + c.cy);
        w[0] = make_float4(xc.x, xc.y, yc.x, yc.y);
        const float2 a1 = split((o.mcn * o.ua[0] - mua * o.n[0]) * (ix * isa));
        const float2 a2 = split((o.mcn * o.ua[1] - mua * o.n[1]) * (iy * isa));
        w[1] = make_float4(a1.x, a1.y, a2.x, a2.y);
        const float2 b1 = split((o.mcn * o.ub[0] - mub * o.n[0]) * (ix * isb));
        const float2 b2 = split((o.mcn * o.ub[1] - mub * o.n[1]) * (iy * isb));
        w[2] = make_float4(b1.x, b1.y, b2.x, b2.y);
        const float2 d1 = split(o.n[0] * ix), d2 = split(o.n[1] * iy);
        const float2 z = split(o.mc[2]);
        // the centre's position is rounded by 2^-48 of it, n . d_centre by a few 2^-53 of its terms
        const float X = fabsf(xc.x), Y = fabsf(yc.x), G = (1.0f + fabsf((xc.x - c.cx) / c.fx) + fabsf((yc.x - c.cy) / c.fy)) * fabsf((float)iD);
        const float err = 0x1p-48f * (fabsf(d1.x) * X + fabsf(d2.x) * Y) + 0x1p-50f * G +
                          0x1p-56f * ((fabsf(a1.x) + fabsf(b1.x)) * X + (fabsf(a2.x) + fabsf(b2.x)) * Y);
        // (a splat whose binary32 decisions that could reach is left to FP64 altogether, like one whose
        // coefficients are not finite)
        w[3] = make_float4(err < 0x1p-34f ? d1.x : __int_as_float(0x7fffffff), d1.y, d2.x, d2.y);
        w[4] = make_float4(z.x, z.y, ax.sigma, err);
    }
}

// The FP64 test of Gaussian g at the pixel centre (px, py).
__device__ __noinline__ bool splat_exact(const SplatSrc &s, const CamDev &c, uint32_t g, float px, float py, float &t,
                                         float &a) {
    const SplatSlot o = splat_in_view(splat_axes(s, g), c);
    return splat_hit(o, c, s.trunc, (double)px, (double)py, t, a);
}

// Binary32 decision at the offset (dx, dy): 1 hit, 0 miss, -1 left to FP64.  Every comparison
// with a value that is not finite fails, which leaves the case to FP64.
__device__ __forceinline__ int splat_decide(const float4 &A, const float4 &B, const float4 &Dc, float Zc, float znear,
                                            float r2, float dx, float dy) {
    constexpr float kU = 32.0f * 0x1p-24f;
    const float p0 = A.x * dx, p1 = A.z * dy, q0 = B.x * dx, q1 = B.z * dy, e0 = Dc.x * dx, e1 = Dc.z * dy;
    const float Nu = p0 + p1, Nv = q0 + q1, D = 1.0f + (e0 + e1);
    const float Mu = fabsf(p0) + fabsf(p1), Mv = fabsf(q0) + fabsf(q1), MD = 1.0f + (fabsf(e0) + fabsf(e1));
    const float f = Nu * Nu + Nv * Nv - r2 * (D * D);
    const float E = kU * (Mu * Mu + Mv * Mv + r2 * (MD * MD));
    if (!(D > 0.001f * MD && Zc > 1.001f * znear * D)) return -1;
    if (f > E) return 0;
    if (f < -E) return 1;
    return -1;
}

// exp(x) of a double-float x in [-4, 0], as a double-float, to about 2^-30: Cody and Waite's reduction
// x = n ln 2 + r with ln 2 in two parts, and the Taylor series of exp(r) with its first three terms in double-float.
__device__ __forceinline__ dfl df_exp(dfl x) {
    constexpr float kLn2h = 0.693145751953125f;                                   // 15 bits: n kLn2h is exact
    constexpr float kLn2l = (float)(0.69314718055994530942 - 0.693145751953125);
    const float n = rintf(x.h * 1.44269504f);
    const dfl r = df_fast_two_sum(fmaf(-n, kLn2h, x.h), fmaf(-n, kLn2l, x.l));
    const dfl r2 = df_two_prod(r.h, r.h);
    float p = 1.0f / 40320.0f;
    p = fmaf(p, r.h, 1.0f / 5040.0f);
    p = fmaf(p, r.h, 1.0f / 720.0f);
    p = fmaf(p, r.h, 1.0f / 120.0f);
    p = fmaf(p, r.h, 1.0f / 24.0f);
    p = fmaf(p, r.h, 1.0f / 6.0f);
    const float low = fmaf(r2.h * r.h, p, fmaf(r.h, r.l, fmaf(0.5f, r2.l, r.l)));
    const dfl s1 = df_two_sum(1.0f, r.h), s2 = df_two_sum(s1.h, 0.5f * r2.h);
    const dfl e = df_fast_two_sum(s2.h, __fadd_rn(__fadd_rn(s1.l, s2.l), low));
    const float sc = __int_as_float((127 + (int)n) << 23);
    return dfl{e.h * sc, e.l * sc};
}

// Depth key and opacity of a hit; false where they are left to FP64.
__device__ __forceinline__ bool splat_values(const float4 &c, const float4 &A, const float4 &B, const float4 &Dc,
                                             const float4 &Z, float px, float py, float &t, float &al) {
    const dfl dx = df_add_f(df_two_sum(px, -c.x), -c.y), dy = df_add_f(df_two_sum(py, -c.z), -c.w);
    const dfl p0 = df_mul(dfl{A.x, A.y}, dx), p1 = df_mul(dfl{A.z, A.w}, dy), Nu = df_add_fast(p0, p1);
    const dfl q0 = df_mul(dfl{B.x, B.y}, dx), q1 = df_mul(dfl{B.z, B.w}, dy), Nv = df_add_fast(q0, q1);
    const dfl e0 = df_mul(dfl{Dc.x, Dc.y}, dx), e1 = df_mul(dfl{Dc.z, Dc.w}, dy);
    const dfl D = df_add_f(df_add_fast(e0, e1), 1.0f);
    const dfl tt = df_div_rcp(dfl{Z.x, Z.y}, D);
    const dfl q = df_div_rcp(df_add_fast(df_mul(Nu, Nu), df_mul(Nv, Nv)), df_mul(D, D));
    const dfl a = df_mul_f(df_exp(dfl{-0.5f * q.h, -0.5f * q.l}), Z.z);
    t = tt.h;
    al = __fadd_rn(a.h, a.l);
    // errors: of D at most err; of Nu and Nv together 2^8 err; so of t err / D, of q 1400 err / D (q < 8)
    const float err = Z.w + 0x1p-44f * (1.0f + fabsf(e0.h) + fabsf(e1.h)) +
                      0x1p-52f * ((fabsf(p0.h) + fabsf(p1.h)) + (fabsf(q0.h) + fabsf(q1.h)));
    // tt.h is the rounding of the depth unless its low part reaches half a unit of tt.h
    const uint32_t tb = __float_as_uint(tt.h);
    const float half = __uint_as_float(tb & 0x7f800000u) * 0x1p-24f;
    return err < 0x1p-40f * D.h && (tb & 0x007fffffu) != 0u &&
           fabsf(tt.l) * D.h < half * D.h - tt.h * fmaf(D.h, 0x1p-45f, err) && q.h < 8.0f && q.h >= 0.0f;
}

// Pixel rectangle of a polygon (decided vertices dv) clipped to the tile, as pair_geo; 0 if empty. (Far from
// the origin the vertices of a small splat may round to one point: its centres are found within the pad.)
__device__ __forceinline__ uint32_t polygon_geo(const float4 *__restrict__ dv, int W, int H, int tx0, int ty0, int tx1,
                                                int ty1) {
    constexpr int K = kSplatK;
    float x[K + 1], y[K + 1];
    uint32_t vmask = 0;
    float ox = 0.0f, oy = 0.0f, pad = 0.0f;
#pragma unroll
    for (int k = 0; k <= K; ++k) {
        const float4 d = __ldg(dv + k);
        x[k] = d.x;
        y[k] = d.y;
        if (d.z > 0.0f) vmask |= 1u << k;   // binning marks invalid vertices with Z = -1
        if (k == 0) ox = d.w;
        if (k == 1) oy = d.w;
        if (k == 2) pad = d.w;
    }
    const uint32_t tmask = tri_valid_mask(vmask, K);
    if (tmask == 0) return 0;
    float mnx = 3.0e38f, mxx = -3.0e38f, mny = 3.0e38f, mxy = -3.0e38f;
#pragma unroll
    for (int k = 0; k <= K; ++k) {
        if (!vertex_used(tmask, k, K)) continue;
        mnx = fminf(mnx, x[k]); mxx = fmaxf(mxx, x[k]);
        mny = fminf(mny, y[k]); mxy = fmaxf(mxy, y[k]);
    }
    const FanRect r = rect_from_bounds_rel(mnx - pad, mxx + pad, mny - pad, mxy + pad, (int)ox, (int)oy, W, H);
    if (r.empty) return 0;
    const int x0 = max(r.i0, tx0), x1 = min(r.i1, tx1), y0 = max(r.j0, ty0), y1 = min(r.j1, ty1);
    if (x0 > x1 || y0 > y1) return 0;
    return pair_geo(x0 - tx0, y0 - ty0, x1 - x0 + 1, y1 - y0 + 1);
}

template <int TILE, bool FILL>
struct SplatMem {
    float4 c[32], A[32], B[32], D[32], Z[32];   // staged coefficients
    float4 col[FILL ? 32 : 1];                  // colour, Gaussian id (bits)
    uint2 info[32];                             // first index in the packed space, rectangle
    uint32_t gid[32];
    uint32_t cnt[TILE * TILE];                  // fragments so far, or next record of each pixel
    uint32_t fits[FILL ? 32 : 1];               // pixels whose records fit the buffer
    uint2 ring[FILL ? 64 : 1];
};

// (14 blocks: the FP64 test's registers spill instead of halving the warps in flight; it is rare)
template <int TILE, bool FILL>
__device__ __forceinline__ void splat_item(const SplatArgs &a, char *smem, uint32_t item) {
    using Mem = SplatMem<TILE, FILL>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Mem &S = reinterpret_cast<Mem *>(smem)[warp];
    const uint4 it = a.items[item];
    const int view = view_of_tile(a.vt, it.x);
    const ViewDev &vw = a.vt.v[view];
    const CamDev &cam = vw.cam;
    const int tile = (int)(it.x - vw.tile_base), tiles_x = (int)vw.tiles_x;
    const int tx0 = (tile % tiles_x) * TILE, ty0 = (tile / tiles_x) * TILE;
    const int tx1 = min(tx0 + TILE, cam.width) - 1, ty1 = min(ty0 + TILE, cam.height) - 1;
    uint32_t *icnt = a.icnt + (size_t)item * TILE * TILE;
    bool all_fit = true;
    for (int i = lane; i < TILE * TILE; i += 32) {
        uint32_t b = 0;
        bool fit = true;
        const int x = tx0 + (i % TILE), y = ty0 + (i / TILE);
        if (FILL && x <= tx1 && y <= ty1) {
            const size_t pix = vw.pix_base + (size_t)y * cam.width + x;
            const uint32_t o = a.offsets[pix];
            // a pixel whose records would not fit gets none (the overflow is reported)
            fit = (int64_t)o + a.counts[pix] <= a.frag_cap;
            b = o + icnt[i];
        }
        S.cnt[i] = b;
        if (FILL) {
            const uint32_t m = __ballot_sync(0xffffffffu, fit);
            if (lane == 0) S.fits[i >> 5] = m;
            all_fit = all_fit && m == 0xffffffffu;
        }
    }
    const uint32_t lt = (1u << lane) - 1u, le = 0xffffffffu >> (31 - lane);
    uint32_t head = 0, queued = 0, n_test = 0;
    for (uint32_t cb = it.y; cb < it.z; cb += 32) {
        const bool mine = cb + lane < it.z;
        const uint32_t g = mine ? __ldg(a.list + cb + lane) : 0u;
        uint32_t geo = 0;
        if (mine)
            geo = FILL ? a.pinfo[cb + lane].y
                       : polygon_geo(a.dec + (size_t)view * (size_t)a.V + (size_t)g * (kSplatK + 1), cam.width,
                                     cam.height, tx0, ty0, tx1, ty1);
        const uint32_t n_mine = geo ? (((geo >> 12) & 63u) + 1u) * (((geo >> 18) & 63u) + 1u) : 0u;
        const bool in = n_mine != 0u;
        const uint32_t live = __ballot_sync(0xffffffffu, in);
        const int slot = __popc(live & lt);
        uint32_t excl = n_mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, excl, o);
            if (lane >= o) excl += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, excl, 31);
        excl -= n_mine;
        __syncwarp();   // the previous pairs are done with the stage
        if (in) {
            const float4 *w = a.coef + 5 * ((size_t)view * (size_t)a.N + g);
            S.c[slot] = __ldg(w);
            S.A[slot] = __ldg(w + 1);
            S.B[slot] = __ldg(w + 2);
            S.D[slot] = __ldg(w + 3);
            S.Z[slot] = __ldg(w + 4);
            if (FILL) {
                const float *col = a.spl.rgb + 3 * (size_t)g;
                S.col[slot] = make_float4(__ldg(col), __ldg(col + 1), __ldg(col + 2), 0.0f);
            }
            S.info[slot] = make_uint2(excl, geo);
            S.gid[slot] = g;
        }
        __syncwarp();
        uint32_t hit_slots = 0;
        for (uint32_t base = 0; base < total; base += 32) {
            // the splats' indices start one after another: an index belongs to the last that
            // starts at or before it
            const int before = __popc(__ballot_sync(0xffffffffu, in && excl < base));
            const uint32_t here = in && excl >= base && excl < base + 32 ? 1u << (excl - base) : 0u;
            const uint32_t starts = __reduce_or_sync(0xffffffffu, here);
            const int f = before + __popc(starts & le) - 1;
            const uint32_t idx = base + lane;
            uint32_t x = 0, y = 0;
            int hit = 0, lp = -1;
            if (idx < total) {
                ++n_test;
                const uint2 inf = S.info[f];
                const uint32_t local = idx - inf.x, w = ((inf.y >> 12) & 63u) + 1u;
                // (local + 0.5) / w is at least 1/(2w) away from an integer: exact row
                const uint32_t yy = (uint32_t)__fdividef((float)local + 0.5f, (float)w);
                x = (inf.y & 63u) + (local - yy * w);
                y = ((inf.y >> 6) & 63u) + yy;
                const float px = (float)(tx0 + (int)x) + 0.5f, py = (float)(ty0 + (int)y) + 0.5f;
                const float4 c = S.c[f];
                hit = splat_decide(S.A[f], S.B[f], S.D[f], S.Z[f].x, cam.znear, a.r2, __fsub_rn(px, c.x) - c.y,
                                   __fsub_rn(py, c.z) - c.w);
                if (hit < 0) {
                    float t, al;
                    hit = splat_exact(a.spl, cam, S.gid[f], px, py, t, al) ? 1 : 0;
                }
                if (hit) lp = (int)(y * TILE + x);
            }
            if (!FILL) {   // counting: the order of a pixel's slots does not matter yet
                hit_slots |= __reduce_or_sync(0xffffffffu, hit ? 1u << f : 0u);
                if (hit) atomicAdd(&S.cnt[lp], 1u);
                continue;
            }
            // (a pixel's records may come in any order: the resolve sorts them)
            uint32_t rec = 0;
            if (hit && !all_fit && !((S.fits[lp >> 5] >> (lp & 31)) & 1u)) hit = 0;
            if (hit) rec = atomicAdd(&S.cnt[lp], 1u);
            const uint32_t pend = __ballot_sync(0xffffffffu, hit != 0);
            if (hit) S.ring[(head + queued + __popc(pend & lt)) & 63u] = make_uint2((uint32_t)f | x << 5 | y << 10, rec);
            queued += __popc(pend);
            __syncwarp();
            // whole warps of hits, and what is left once these splats' centres are done
            while (queued >= 32u || (queued && base + 32 >= total)) {
                const uint32_t nj = min(queued, 32u);
                if (lane < nj) {
                    const uint2 job = S.ring[(head + lane) & 63u];
                    const int jf = (int)(job.x & 31u);
                    const float px = (float)(tx0 + (int)((job.x >> 5) & 31u)) + 0.5f;
                    const float py = (float)(ty0 + (int)((job.x >> 10) & 31u)) + 0.5f;
                    const float4 Z = S.Z[jf];
                    float t, al;
                    if (!splat_values(S.c[jf], S.A[jf], S.B[jf], S.D[jf], Z, px, py, t, al))
                        splat_exact(a.spl, cam, S.gid[jf], px, py, t, al);
                    const float4 col = S.col[jf];
                    float4 *out = a.frags + (size_t)kRecFwd * (size_t)job.y;
                    st_rec(out, make_float4(t, __uint_as_float(S.gid[jf]), 0.0f, 0.0f), make_float4(col.x, col.y, col.z, al));
                }
                head += nj;
                queued -= nj;
                __syncwarp();
            }
        }
        // each pair's rectangle if it covers any pixel centre
        if (!FILL && mine) a.pinfo[cb + lane] = make_uint2(0u, in && ((hit_slots >> slot) & 1u) ? geo : 0u);
    }
    if (!FILL) {
        __syncwarp();
        for (int i = lane; i < TILE * TILE; i += 32) {
            const uint32_t c = S.cnt[i];   // (nonzero only inside the image)
            if (c)
                icnt[i] = atomicAdd(a.counts + vw.pix_base + (size_t)(ty0 + i / TILE) * cam.width + (size_t)(tx0 + i % TILE), c);
        }
        const unsigned r0 = __reduce_add_sync(0xffffffffu, n_test);
        if (lane == 0) atomicAdd(a.tests + item % kMaskRegions, (unsigned long long)r0);
    }
}

template <int TILE, bool FILL, bool STRIDED>
__global__ void __launch_bounds__(kSplatWarps * 32, 14) splat_raster_kernel(const __grid_constant__ SplatArgs a) {
    extern __shared__ __align__(16) char smem[];
    const uint32_t n_items = a.st->n_items;
    uint32_t item = blockIdx.x * kSplatWarps + threadIdx.x / 32;   // (whole warps: nothing synchronises the block)
    if (!STRIDED) {
        if (item < n_items) splat_item<TILE, FILL>(a, smem, item);
    } else {
        for (; item < n_items; item += gridDim.x * kSplatWarps) {
            splat_item<TILE, FILL>(a, smem, item);
            __syncwarp();   // the stage is free again
        }
    }
}

template <int TILE, bool FILL>
cudaError_t launch_t(const SplatArgs &sa, int64_t max_items, cudaStream_t st) {
    const size_t smem = kSplatWarps * sizeof(SplatMem<TILE, FILL>);
    const int64_t blocks = (max_items + kSplatWarps - 1) / kSplatWarps;
    const bool strided = blocks > kItemBlocks;
    auto fn = strided ? splat_raster_kernel<TILE, FILL, true> : splat_raster_kernel<TILE, FILL, false>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    fn<<<(unsigned)(strided ? kStrideBlocks : blocks), kSplatWarps * 32, smem, st>>>(sa);
    return cudaGetLastError();
}

template <bool FILL>
cudaError_t launch(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    if (L.n_tiles == 0) return cudaSuccess;
    SplatArgs a;
    a.vt = ra.vt;
    a.spl = ra.spl;
    a.N = ra.n_fans;
    a.list = reinterpret_cast<const uint32_t *>(ra.ws + L.off_list);
    a.items = reinterpret_cast<const uint4 *>(ra.ws + L.off_items);
    a.icnt = reinterpret_cast<uint32_t *>(ra.ws + L.off_icnt);
    a.offsets = reinterpret_cast<const uint32_t *>(ra.ws + L.off_offsets);
    a.counts = reinterpret_cast<uint32_t *>(ra.ws + L.off_counts);
    a.frags = reinterpret_cast<float4 *>(ra.ws + L.off_frags);
    a.frag_cap = L.frag_cap;
    a.st = reinterpret_cast<Status *>(ra.ws + L.off_status);
    a.dec = reinterpret_cast<const float4 *>(ra.ws + L.off_dec);
    a.V = L.V;
    a.tests = reinterpret_cast<unsigned long long *>(ra.ws + L.off_mask_cursor);
    a.pinfo = reinterpret_cast<uint2 *>(ra.ws + L.off_maskoff);
    a.coef = ra.splat_coef;
    a.r2 = (float)(ra.spl.trunc * ra.spl.trunc);
    const cudaError_t e = L.tile == 8    ? launch_t<8, FILL>(a, L.max_items, st)
                          : L.tile == 32 ? launch_t<32, FILL>(a, L.max_items, st)
                                         : launch_t<16, FILL>(a, L.max_items, st);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

}  // namespace

size_t splat_coef_bytes(int64_t N, int n_views) { return (size_t)80 * (size_t)N * (size_t)n_views; }

cudaError_t launch_splat_setup(const RenderArgs &ra, cudaStream_t st) {
    if (ra.n_fans == 0) return cudaSuccess;
    splat_setup_kernel<<<(unsigned)((ra.n_fans + kSetupThreads - 1) / kSetupThreads), kSetupThreads, 0, st>>>(
        ra.spl, ra.n_fans, ra.vt, ra.splat_coef);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_splat_count(const RenderArgs &ra, cudaStream_t st) { return launch<false>(ra, st); }
cudaError_t launch_splat_fill(const RenderArgs &ra, cudaStream_t st) { return launch<true>(ra, st); }

}  // namespace ms
