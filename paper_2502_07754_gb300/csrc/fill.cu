// Fill pass of the tile rasterisation: one 32-byte record per fragment -- depth (high),
// triangle id, 0, depth (low), colour, opacity -- at its pixel's offset + the item's slot +
// running index.  It walks the same work items as the count pass (raster.cu), whose coverage
// masks and rectangles say which centres each pair covers.
//
// One warp takes one item (at most kItemFans fans of one tile):
//  1. pairs that cover no centre drop out; the others, kFillFans at a time, are staged with
//     all lanes: one lane a fan for the centre's double-float projection, then one lane a
//     (fan, boundary vertex) for the vertices' screen and view offsets, 1 / depth, colour and
//     opacity;
//  2. the staged fans' rectangles form one packed (fan, pixel) index space, a lane a centre:
//     it reads the centre's mask and takes record slots for its triangles (a pixel's records may
//     come in any order: the resolve sorts them);
//  3. every covered (fan, triangle, centre) goes into a ring of jobs, and whole warps of jobs
//     compute their fragment: perspective-correct barycentrics, values, and the exact-order
//     depth in double-float.
// What bounds it: issue slots (64% of cycles) and the waits of a pair's dependent loads.  Staging with
// every lane and computing fragments 32 at a time, against four lanes a fan and the lanes whose test hit,
// with full groups of fans: 1M fans at 1080p (10.4M fragments) 0.62 -> 0.43 ms, 200k fans at 800x800 0.31 ->
// 0.195 ms, 3M fans in 16 views (42M pairs, 51M fragments) 9.9 -> 4.3 ms (with the strided launch).
#include "raster_common.cuh"

namespace ms {

namespace {

struct FillArgs {
    const float *xyz, *rgb, *alpha;
    int K;
    ViewTable vt;
    const uint32_t *list;             // fans in tile order
    const uint4 *items;               // (tile, start, end, index within tile)
    const uint32_t *icnt;             // [item][tile pixels]: first slot within the pixel
    const uint32_t *offsets, *counts;
    float4 *frags;
    int64_t frag_cap;
    const Status *st;
    const float4 *dec;                // [view][vertex] decided vertices (pairs without stored masks)
    int64_t V;
    const uint32_t *face_mask;        // per fan, bit j = face j drawn; NULL = all
    const uint2 *pinfo;               // per pair: first coverage mask (~0: none stored), rectangle (0: covers nothing)
    const uint16_t *masks;
};

constexpr int kFillWarps = 2;    // warps (work items) per block: items differ widely in cost
// Fans staged together: many where a pair has few centres (8-pixel tiles; 16 views of 3M fans: 18.7 ms with 16,
// 20.1 with 8), else few, for the shared memory of more warps (200k fans at 800x800: 889 us with 16, 869 with 8).
template <int TILE>
constexpr int kFillFans = TILE == 8 ? 16 : 8;

// Words of one warp.  Arrays of one 16-byte word per fan or vertex, so that a job's loads are
// few and its lanes, on fans in any order, spread over the banks.
template <int TILE>
struct FillMem {
    uint32_t *next;      // [TILE^2] next record of each pixel
    uint32_t *fits;      // [TILE^2 / 32] pixels whose records fit the buffer
    uint2 *ring;         // [64] jobs: fan slot | triangle << 4 | x << 8 | y << 13, record
    uint8_t *live;       // [kItemFans] the item's pairs that cover a centre
    uint4 *info;         // [kFillFans<TILE>] first index in the packed space, first mask, rectangle, fan id
    float4 *m;           // [kFillFans<TILE>] centre position, its 1 / depth
    float4 *P;           // [kFillFans<TILE>] view position of the centre (high parts), 0
    float4 *c;           // [kFillFans<TILE>] double-float screen position of the centre (x, then y)
    float4 *pc;          // [kFillFans<TILE>] fx X_c, fy Y_c in double-float
    float4 *zc;          // [kFillFans<TILE>] Z_c in double-float, fan id (bits), 0
    float4 *col;         // [kFillFans<TILE>] the centre's colour and opacity
    float4 *va;          // [kFillFans<TILE>][K] screen offset du, dv, 1 / depth, opacity
    float4 *vb;          // [kFillFans<TILE>][K] view offset x, y in double-float
    float4 *vc;          // [kFillFans<TILE>][K] view offset z in double-float, red, green
    float *vd;           // [kFillFans<TILE>][K] blue
};

template <int TILE>
__host__ __device__ constexpr size_t fill_warp_bytes(int K) {
    return (size_t)TILE * TILE * 4 + 32 * 4 + 64 * 8 + kItemFans + (size_t)kFillFans<TILE> * (7 * 16 + (size_t)K * 52);
}

template <int TILE>
__device__ __forceinline__ FillMem<TILE> fill_mem(char *p, int K) {
    FillMem<TILE> s;
    s.next = reinterpret_cast<uint32_t *>(p);
    s.fits = s.next + TILE * TILE;
    s.ring = reinterpret_cast<uint2 *>(s.fits + 32);
    s.live = reinterpret_cast<uint8_t *>(s.ring + 64);
    s.info = reinterpret_cast<uint4 *>(s.live + kItemFans);
    s.m = reinterpret_cast<float4 *>(s.info + kFillFans<TILE>);
    s.P = s.m + kFillFans<TILE>;
    s.c = s.P + kFillFans<TILE>;
    s.pc = s.c + kFillFans<TILE>;
    s.zc = s.pc + kFillFans<TILE>;
    s.col = s.zc + kFillFans<TILE>;
    s.va = s.col + kFillFans<TILE>;
    s.vb = s.va + kFillFans<TILE> * K;
    s.vc = s.vb + kFillFans<TILE> * K;
    s.vd = reinterpret_cast<float *>(s.vc + kFillFans<TILE> * K);
    return s;
}

// Depth of triangle (c, b_j, b_j+1) at the pixel centre (pxc, pyc) (absolute screen
// coordinates), in double-float: the view depth where the pixel's ray
// r = ((x - cx) / fx, (y - cy) / fy, 1) meets the triangle's plane, Z = n . P_c / n . r with
// n = e1 x e2 the normal from the vertices' exact view offsets and P_c the centre's
// view position (numerator and denominator both scaled by fx fy: xf, yf, zc), which equals
// 1 / sum_k (lambda_k / Z_k) of the perspective-correct barycentrics.  Clamped to the
// triangle's vertex depths, where a covered centre lies (the clamp acts only where the
// decided coverage and the exact plane differ by rounding; a ray parallel to the plane
// takes the least vertex depth).
__device__ __forceinline__ dfl frag_depth_df(const DfVec &e1, const DfVec &e2, dfl xf, dfl yf, dfl zc, float pxc,
                                             float pyc, const CamDev &c) {
    const dfl nx = df_add_fast(df_mul(e1.y, e2.z), df_neg(df_mul(e1.z, e2.y)));
    const dfl ny = df_add_fast(df_mul(e1.z, e2.x), df_neg(df_mul(e1.x, e2.z)));
    const dfl nz = df_add_fast(df_mul(e1.x, e2.y), df_neg(df_mul(e1.y, e2.x)));
    const dfl pa = df_mul_f(nx, c.fy), pb = df_mul_f(ny, c.fx), pn = df_mul_f(df_mul_f(nz, c.fx), c.fy);
    const dfl num = df_add_fast(df_add_fast(df_mul(pa, xf), df_mul(pb, yf)), df_mul(pn, zc));
    const dfl den = df_add_fast(df_add_fast(df_mul(pa, df_two_sum(pxc, -c.cx)), df_mul(pb, df_two_sum(pyc, -c.cy))),
                                pn);
    const dfl z1 = df_add_fast(zc, e1.z), z2 = df_add_fast(zc, e2.z);
    dfl lo = zc, hi = zc;
    if (df_lt(z1, lo)) lo = z1;
    if (df_lt(z2, lo)) lo = z2;
    if (df_lt(hi, z1)) hi = z1;
    if (df_lt(hi, z2)) hi = z2;
    if (den.h == 0.0f) return lo;
    dfl z = df_div_rcp(num, den);
    if (!(z.h == z.h)) return lo;   // NaN
    if (df_lt(z, lo)) z = lo;
    if (df_lt(hi, z)) z = hi;
    return z;
}

// Coverage of the pixel (px, py) by a fan whose masks did not fit the mask buffer, straight
// from its decided vertices dv: the same edge values and tie rules as cover_mask, triangle by
// triangle.
__device__ __noinline__ uint32_t cover_direct(const float4 *__restrict__ dv, int K, uint32_t drawn, int px, int py) {
    auto tie = [](float ex, float ey) { return ey < 0.0f || (ey == 0.0f && ex > 0.0f); };
    const float4 c = __ldg(dv), b0 = __ldg(dv + 1);
    const float pxc = (float)(px - (int)c.w) + 0.5f, pyc = (float)(py - (int)b0.w) + 0.5f;
    const float qx = __fsub_rn(pxc, c.x), qy = __fsub_rn(pyc, c.y);
    uint32_t hits = 0;
    float4 b = b0;
    for (int j = 0; j < K; ++j) {
        const bool wrap = j + 1 == K;
        const float4 n = wrap ? b0 : __ldg(dv + 2 + j);
        if (c.z > 0.0f && b.z > 0.0f && n.z > 0.0f && ((drawn >> j) & 1u)) {
            const float ar = dec_area2(c.x, c.y, b.x, b.y, n.x, n.y);
            const bool neg = ar < 0.0f;
            const float sx = __fsub_rn(b.x, c.x), sy = __fsub_rn(b.y, c.y);
            const float tx = __fsub_rn(n.x, c.x), ty = __fsub_rn(n.y, c.y);
            const float S = __fsub_rn(__fmul_rn(sx, qy), __fmul_rn(sy, qx));
            const float T = __fsub_rn(__fmul_rn(tx, qy), __fmul_rn(ty, qx));
            const float Sf = neg ? -S : S, Tf = neg ? T : -T;   // both positive inside
            const bool okS = Sf > 0.0f || (S == 0.0f && (neg ? tie(-sx, -sy) : tie(sx, sy)));
            const bool okT = Tf > 0.0f || (T == 0.0f && (neg ? tie(tx, ty) : tie(-tx, -ty)));
            const float rx = wrap ? __fsub_rn(b.x, n.x) : __fsub_rn(n.x, b.x);
            const float ry = wrap ? __fsub_rn(b.y, n.y) : __fsub_rn(n.y, b.y);
            const float Rc = dec_edge(rx, ry, wrap ? n.x : b.x, wrap ? n.y : b.y, pxc, pyc);
            const bool flip = wrap != neg;
            const float E0 = flip ? -Rc : Rc;
            const bool okR = E0 > 0.0f || (E0 == 0.0f && (flip ? tie(-rx, -ry) : tie(rx, ry)));
            if (ar != 0.0f && okS && okT && okR) hits |= 1u << j;
        }
        b = n;
    }
    return hits;
}

template <int TILE, int KT>
__device__ __forceinline__ void fill_item(const FillArgs &a, char *smem, uint32_t item) {
    const int K = KT > 0 ? KT : a.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint4 it = a.items[item];
    const int view = view_of_tile(a.vt, it.x);
    const ViewDev &vw = a.vt.v[view];
    const CamDev &cam = vw.cam;
    const int tile = (int)(it.x - vw.tile_base), tiles_x = (int)vw.tiles_x;
    const int tx0 = (tile % tiles_x) * TILE, ty0 = (tile / tiles_x) * TILE;
    const FillMem<TILE> S = fill_mem<TILE>(smem + (size_t)warp * fill_warp_bytes<TILE>(K), K);
    bool all_fit = true;
    {
        const int tx1 = min(tx0 + TILE, cam.width) - 1, ty1 = min(ty0 + TILE, cam.height) - 1;
        const uint32_t *icnt = a.icnt + (size_t)item * TILE * TILE;
        for (int i = lane; i < TILE * TILE; i += 32) {
            const int x = tx0 + (i % TILE), y = ty0 + (i / TILE);
            uint32_t b = 0;
            bool fit = true;
            if (x <= tx1 && y <= ty1) {
                const size_t pix = vw.pix_base + (size_t)y * cam.width + x;
                const uint32_t o = a.offsets[pix];
                // a pixel whose records would not fit gets none (the overflow is reported)
                fit = (int64_t)o + a.counts[pix] <= a.frag_cap;
                b = o + icnt[i];
            }
            S.next[i] = b;
            const uint32_t f = __ballot_sync(0xffffffffu, fit);
            if (lane == 0) S.fits[i >> 5] = f;
            all_fit = all_fit && f == 0xffffffffu;
        }
    }
    const uint32_t lt = (1u << lane) - 1u, le = 0xffffffffu >> (31 - lane);
    uint32_t head = 0, queued = 0;   // the ring
    // the pairs that cover a pixel centre, by their place in the item
    int n_live = 0;
    for (uint32_t cb = it.y; cb < it.z; cb += 32) {
        const bool covers = cb + lane < it.z && __ldg(&a.pinfo[cb + lane].y) != 0u;
        const uint32_t live = __ballot_sync(0xffffffffu, covers);
        if (covers) S.live[n_live + __popc(live & lt)] = (uint8_t)(cb - it.y + lane);
        n_live += __popc(live);
    }
    for (int l0 = 0; l0 < n_live; l0 += kFillFans<TILE>) {
        const int nl = min(kFillFans<TILE>, n_live - l0), slot = lane;
        const bool in = lane < nl;
        __syncwarp();   // the list is written, the previous fans' jobs are done
        uint2 pinf = make_uint2(0u, 0u);
        uint32_t fan = 0, excl = 0;
        if (in) {
            const uint32_t at = it.y + S.live[l0 + lane];
            pinf = __ldg(a.pinfo + at);
            fan = __ldg(a.list + at);
            excl = (((pinf.y >> 12) & 63u) + 1u) * (((pinf.y >> 18) & 63u) + 1u);
        }
        const uint32_t n_mine = excl;
#pragma unroll
        for (int o = 1; o < kFillFans<TILE>; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, excl, o);
            if (lane >= o) excl += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, excl, kFillFans<TILE> - 1);
        excl -= n_mine;
        if (in) {
            const float *p = a.xyz + (size_t)fan * (K + 1) * 3;
            const float m[3] = {__ldg(p), __ldg(p + 1), __ldg(p + 2)};
            const float *col = a.rgb + (size_t)fan * (K + 1) * 3;
            S.col[slot] = make_float4(__ldg(col), __ldg(col + 1), __ldg(col + 2),
                                      __ldg(a.alpha + (size_t)fan * (K + 1)));
            const CentreProj cp = project_centre(cam, m);
            const dfl zc = df_fast_two_sum(cp.Zh, cp.Zl);
            const dfl xf = df_mul_f(df_fast_two_sum(cp.Xh, cp.Xl), cam.fx);
            const dfl yf = df_mul_f(df_fast_two_sum(cp.Yh, cp.Yl), cam.fy);
            S.info[slot] = make_uint4(excl, pinf.x, pinf.y, fan);
            S.m[slot] = make_float4(m[0], m[1], m[2], 1.0f / zc.h);
            S.P[slot] = make_float4(cp.Xh, cp.Yh, cp.Zh, 0.0f);
            S.c[slot] = make_float4(cp.xh, cp.xl, cp.yh, cp.yl);
            S.pc[slot] = make_float4(xf.h, xf.l, yf.h, yf.l);
            S.zc[slot] = make_float4(zc.h, zc.l, __uint_as_float(fan), 0.0f);
        }
        __syncwarp();
        for (int i = lane; i < nl * K; i += 32) {   // one (fan, boundary vertex) a lane
            const int f = i / K, k = i - f * K;
            const float4 mm = S.m[f], PP = S.P[f], zz = S.zc[f];
            const size_t v = (size_t)__float_as_uint(zz.z) * (K + 1) + 1 + k;
            const float *pi = a.xyz + 3 * v, *col = a.rgb + 3 * v;
            const float r = __ldg(col), g = __ldg(col + 1), b = __ldg(col + 2), al = __ldg(a.alpha + v);
            const float m[3] = {mm.x, mm.y, mm.z};
            const float d[3] = {__ldg(pi) - m[0], __ldg(pi + 1) - m[1], __ldg(pi + 2) - m[2]};
            CentreProj cp;
            cp.Xh = PP.x;
            cp.Yh = PP.y;
            cp.Zh = PP.z;
            float du, dv, X, Y, Z;
            vertex_offset(cam, cp, d, du, dv, X, Y, Z);
            // the exact view offset e = R (b_i - c) in double-float, for the fragment depths
            const DfVec e = df_view_offset(cam, m, pi);
            S.va[i] = make_float4(du, dv, 1.0f / df_add(dfl{zz.x, zz.y}, e.z).h, al);
            S.vb[i] = make_float4(e.x.h, e.x.l, e.y.h, e.y.l);
            S.vc[i] = make_float4(e.z.h, e.z.l, r, g);
            S.vd[i] = b;
        }
        __syncwarp();
        for (uint32_t base = 0; base < total; base += 32) {
            // the fan of each index: the fans start one after another, so an index's fan is the
            // last one that starts at or before it
            const int before = __popc(__ballot_sync(0xffffffffu, in && excl < base));
            const uint32_t here = in && excl >= base && excl < base + 32 ? 1u << (excl - base) : 0u;
            const uint32_t starts = __reduce_or_sync(0xffffffffu, here);
            const int f = before + __popc(starts & le) - 1;
            const uint32_t idx = base + lane;
            uint32_t hits = 0, x = 0, y = 0, rec = 0;
            if (idx < total) {
                const uint4 inf = S.info[f];
                const uint32_t local = idx - inf.x, w = ((inf.z >> 12) & 63u) + 1u;
                // (local + 0.5) / w is at least 1/(2w) away from an integer: exact row
                const uint32_t yy = (uint32_t)__fdividef((float)local + 0.5f, (float)w);
                x = (inf.z & 63u) + (local - yy * w);
                y = ((inf.z >> 6) & 63u) + yy;
                if (inf.y != ~0u)
                    hits = __ldg(a.masks + inf.y + local);
                else
                    hits = cover_direct(a.dec + (size_t)view * (size_t)a.V + (size_t)inf.w * (K + 1), K,
                                        a.face_mask ? __ldg(a.face_mask + inf.w) : ~0u, tx0 + (int)x, ty0 + (int)y);
                const uint32_t lp = y * TILE + x;
                if (!all_fit && !((S.fits[lp >> 5] >> (lp & 31u)) & 1u)) hits = 0;
                if (hits) rec = atomicAdd(&S.next[lp], (uint32_t)__popc(hits));
            }
            bool more;
            do {
                const uint32_t pend = __ballot_sync(0xffffffffu, hits != 0u);
                if (hits) {
                    const uint32_t j = (uint32_t)__ffs(hits) - 1u;
                    S.ring[(head + queued + __popc(pend & lt)) & 63u] =
                        make_uint2((uint32_t)f | j << 4 | x << 8 | y << 13, rec);
                    hits &= hits - 1;
                    ++rec;
                }
                queued += __popc(pend);
                more = __any_sync(0xffffffffu, hits != 0u);
                __syncwarp();
                // whole warps of jobs, and what is left once these fans' centres are done
                while (queued >= 32u || (queued && !more && base + 32 >= total)) {
                    const uint32_t nj = min(queued, 32u);
                    if (lane < nj) {
                        const uint2 job = S.ring[(head + lane) & 63u];
                        const int jf = (int)(job.x & 15u), j = (int)((job.x >> 4) & 15u);
                        const float pxc = (float)(tx0 + (int)((job.x >> 8) & 31u)) + 0.5f;
                        const float pyc = (float)(ty0 + (int)((job.x >> 13) & 31u)) + 0.5f;
                        const int vj = jf * K + j, vn = j + 1 == K ? jf * K : vj + 1;
                        const float4 jb = S.vb[vj], jc = S.vc[vj], nb = S.vb[vn], nc = S.vc[vn];
                        const float4 pc = S.pc[jf], zc = S.zc[jf];
                        const DfVec e1 = {{jb.x, jb.y}, {jb.z, jb.w}, {jc.x, jc.y}};
                        const DfVec e2 = {{nb.x, nb.y}, {nb.z, nb.w}, {nc.x, nc.y}};
                        const dfl zf = frag_depth_df(e1, e2, dfl{pc.x, pc.y}, dfl{pc.z, pc.w}, dfl{zc.x, zc.y}, pxc,
                                                     pyc, cam);
                        // perspective-correct barycentrics from the accurate centre offsets
                        const float4 c = S.c[jf], ja = S.va[vj], na = S.va[vn], cc = S.col[jf];
                        const float izc = S.m[jf].w, izj = ja.z, izn = na.z;
                        const float ox = __fsub_rn(c.x, pxc) + c.y;
                        const float oy = __fsub_rn(c.z, pyc) + c.w;
                        const float ujx = ox + ja.x, ujy = oy + ja.y;
                        const float unx = ox + na.x, uny = oy + na.y;
                        const float w0 = (ujx * uny - ujy * unx) * izc;
                        const float w1 = (unx * oy - uny * ox) * izj;
                        const float w2 = (ox * ujy - oy * ujx) * izn;
                        const float iW = 1.0f / (w0 + w1 + w2);
                        const float m0 = w0 * iW, m1 = w1 * iW, m2 = w2 * iW;
                        const float al = m0 * cc.w + m1 * ja.w + m2 * na.w;
                        const float c0 = m0 * cc.x + m1 * jc.z + m2 * nc.z;
                        const float c1 = m0 * cc.y + m1 * jc.w + m2 * nc.w;
                        const float c2 = m0 * cc.z + m1 * S.vd[vj] + m2 * S.vd[vn];
                        const uint32_t tri = __float_as_uint(zc.z) * (uint32_t)K + (uint32_t)j;
                        float4 *out = a.frags + (size_t)kRecFwd * (size_t)job.y;
                        out[0] = make_float4(zf.h, __uint_as_float(tri), 0.0f, zf.l);
                        out[1] = make_float4(c0, c1, c2, al);
                    }
                    head += nj;
                    queued -= nj;
                    __syncwarp();
                }
            } while (more);
        }
    }
}

template <int TILE, int KT, bool STRIDED>
__global__ void __launch_bounds__(kFillWarps * 32) fill_kernel(const __grid_constant__ FillArgs a) {
    extern __shared__ __align__(16) char smem[];
    const uint32_t n_items = a.st->n_items;
    uint32_t item = blockIdx.x * kFillWarps + threadIdx.x / 32;   // (whole warps: nothing synchronises the block)
    if (!STRIDED) {
        if (item < n_items) fill_item<TILE, KT>(a, smem, item);
    } else {
        for (; item < n_items; item += gridDim.x * kFillWarps) {
            fill_item<TILE, KT>(a, smem, item);
            __syncwarp();   // the stage is free again
        }
    }
}

template <int TILE, int KT>
cudaError_t launch_t(const FillArgs &fa, int64_t max_items, int K, cudaStream_t st) {
    const size_t smem = kFillWarps * fill_warp_bytes<TILE>(K);
    const int64_t blocks = (max_items + kFillWarps - 1) / kFillWarps;
    const bool strided = blocks > kItemBlocks;
    auto fn = strided ? fill_kernel<TILE, KT, true> : fill_kernel<TILE, KT, false>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    fn<<<(unsigned)(strided ? kStrideBlocks : blocks), kFillWarps * 32, smem, st>>>(fa);
    return cudaGetLastError();
}

template <int TILE>
cudaError_t launch_k(const FillArgs &fa, int64_t max_items, int K, cudaStream_t st) {
    if (K == 8) return launch_t<TILE, 8>(fa, max_items, K, st);
    if (K == 6) return launch_t<TILE, 6>(fa, max_items, K, st);
    return launch_t<TILE, 0>(fa, max_items, K, st);
}

}  // namespace

cudaError_t launch_fill(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    if (L.n_tiles == 0) return cudaSuccess;
    FillArgs a;
    a.xyz = ra.xyz;
    a.rgb = ra.rgb;
    a.alpha = ra.alpha;
    a.K = ra.K;
    a.vt = ra.vt;
    a.list = reinterpret_cast<const uint32_t *>(ra.ws + L.off_list);
    a.items = reinterpret_cast<const uint4 *>(ra.ws + L.off_items);
    a.icnt = reinterpret_cast<const uint32_t *>(ra.ws + L.off_icnt);
    a.offsets = reinterpret_cast<const uint32_t *>(ra.ws + L.off_offsets);
    a.counts = reinterpret_cast<const uint32_t *>(ra.ws + L.off_counts);
    a.frags = reinterpret_cast<float4 *>(ra.ws + L.off_frags);
    a.frag_cap = L.frag_cap;
    a.st = reinterpret_cast<const Status *>(ra.ws + L.off_status);
    a.dec = reinterpret_cast<const float4 *>(ra.ws + L.off_dec);
    a.V = L.V;
    a.face_mask = ra.prm.face_mask;
    a.pinfo = reinterpret_cast<const uint2 *>(ra.ws + L.off_maskoff);
    a.masks = reinterpret_cast<const uint16_t *>(ra.ws + L.off_masks);
    const cudaError_t e = L.tile == 8    ? launch_k<8>(a, L.max_items, ra.K, st)
                          : L.tile == 32 ? launch_k<32>(a, L.max_items, ra.K, st)
                                         : launch_k<16>(a, L.max_items, ra.K, st);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

}  // namespace ms
