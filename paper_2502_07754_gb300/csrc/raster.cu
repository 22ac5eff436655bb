// Tile rasterisation into a per-pixel fragment buffer (A-buffer) in HBM: the count pass.
//
// Every tile's fan list is cut into work items of at most kItemFans fans (tiles.cu); one warp
// rasterises one item, so a hot tile with thousands of fans spreads over many warps instead of
// serialising on one.  A warp takes 32 pairs at a time, a lane a pair: from the fan's decided
// vertices it forms the triangles' spoke and rim directions (to shared memory), their
// orientations and the fan's pixel rectangle inside the tile.  The rectangles' rows, cut into runs
// of two pixels, form one index space, a lane a run: it answers the two (fan, pixel) tests with the
// binary32 decision formulas, sharing the spoke loads and the row's products.  No block barriers
// are used.  What bounds it: issue slots (56 to 70% busy).  Against two lanes
// staging a pair's words one triangle after the other and a lane a test: 200k fans at 800x800 (9M tests)
// 103 -> 78 us, 3M fans in 16 views (42M pairs, 96M tests) 4.3 -> 3.3 ms, and 2.1 ms with the strided launch
//
// The pass leaves the coverage mask of every test, per pair its first mask index and its pixel
// rectangle within the tile (zero when the pair covers no pixel centre, so the fill skips it),
// the pixels' fragment counts, and each item's first slot within every pixel it touches: an
// item adds its count to the pixel's and takes what was there before (a pixel's records may come
// in any order).  pixel_alloc_kernel then gives the pixels their record ranges, and the fill
// pass (fill.cu) walks the same items with the stored masks and rectangles and writes the
// records.
#include <algorithm>

#include "raster_common.cuh"

namespace ms {

namespace {

struct RastArgs {
    int K;
    ViewTable vt;
    const uint32_t *list;      // fans in tile order
    const uint4 *items;        // (tile, start, end, index within tile)
    uint32_t *icnt;            // [item][tile pixels]: first slot within the pixel (where the item has fragments)
    uint32_t *counts;          // fragments of each pixel (zeroed per render)
    Status *st;
    const float4 *dec;         // [view][vertex] decided vertices from binning
    int64_t V;
    const uint32_t *face_mask; // per fan, bit j = face j drawn; NULL = all
    uint2 *pinfo;              // per pair: index of its first coverage mask (~0 if none stored), and its
                               // pixel rectangle clipped to the tile (pair_geo; 0 if empty)
    uint16_t *masks;           // coverage masks (bit j: triangle j) of the tests
    int64_t mask_cap;
    uint32_t mask_regions;
    unsigned long long *mask_cursor;   // [mask_regions] tests of the mask regions (zeroed per render)
};

constexpr int kRastWarps = 2;   // warps (work items) per block: items differ widely in cost

// Words of one warp.
struct CountMem {
    uint32_t *cnt;    // [TILE^2] fragments so far
    float4 *c;        // [32] first pixel centre of the tile and the fan's centre, both relative to the fan's origin
    uint4 *info;      // [32] of the pairs with tests: first run, first test, rectangle, lane of the pair
    uint32_t *flags;  // [32] bits 0..15 valid triangle, 16..31 negative orientation
    float2 *sd;       // [K][32] spoke directions b_i - c
    float4 *rim;      // [K][32] rim directions, lower index to higher, and the lower vertex
};

template <int TILE>
__host__ __device__ constexpr size_t count_warp_bytes(int K) {
    return (size_t)TILE * TILE * 4 + 32 * (16 + 16 + 4 + (size_t)K * 24);
}

template <int TILE>
__device__ __forceinline__ CountMem count_mem(char *p, int K) {
    CountMem s;
    s.cnt = reinterpret_cast<uint32_t *>(p);
    s.c = reinterpret_cast<float4 *>(s.cnt + TILE * TILE);
    s.info = reinterpret_cast<uint4 *>(s.c + 32);
    s.flags = reinterpret_cast<uint32_t *>(s.info + 32);
    s.rim = reinterpret_cast<float4 *>(s.flags + 32);
    s.sd = reinterpret_cast<float2 *>(s.rim + 32 * K);
    return s;
}

// Top-left tie rule: whether a centre exactly on an edge of direction (ex, ey) belongs to it.
__device__ __forceinline__ bool edge_tie(float ex, float ey) { return ey < 0.0f || (ey == 0.0f && ex > 0.0f); }

// Coverage of the pixel centre (pxc, pyc), at (qx, qy) from the fan's centre, by the pair of lane
// f: bit j is set when triangle j covers it, the conjunction of its three edge tests.  N has the sign
// bits of the spoke values S_i (bit i); a spoke's two pass bits, as the edge c -> b_i and as its
// reverse, are these bits and their complement unless a value is zero (`zero`), where the tie rule
// decides.  Only triangles passing both spokes get the rim edge, nearly always one.
template <int KT>
__device__ __forceinline__ uint32_t cover_mask(const CountMem &S, int K, int f, uint32_t flags, uint32_t N, bool zero,
                                               float pxc, float pyc, float qx, float qy) {
    const uint32_t full = (1u << K) - 1u;
    uint32_t P = ~N & full;
    if (zero) {   // a centre on a spoke's line
        P = N = 0;
#pragma unroll 1
        for (int i = 0; i < K; ++i) {
            const float2 d = S.sd[i * 32 + f];
            const float Si = __fsub_rn(__fmul_rn(d.x, qy), __fmul_rn(d.y, qx));
            P |= (uint32_t)(Si > 0.0f || (Si == 0.0f && edge_tie(d.x, d.y))) << i;
            N |= (uint32_t)(Si < 0.0f || (Si == 0.0f && edge_tie(-d.x, -d.y))) << i;
        }
    }
    const uint32_t Pn = ((P >> 1) | (P << (K - 1))) & full;   // bit j: spoke j+1
    const uint32_t Nn = ((N >> 1) | (N << (K - 1))) & full;
    const uint32_t neg = flags >> 16;
    // oriented rim: b_j -> b_{j+1} for positive orientation, reversed otherwise (the stored direction
    // runs from the lower index to the higher, so the last one is reversed already)
    const uint32_t flip = neg ^ (1u << (K - 1));
    uint32_t cand = ((P & Nn & ~neg) | (N & Pn & neg)) & flags & full;
    uint32_t hits = 0;
    while (cand) {
        const int j = __ffs(cand) - 1;
        cand &= cand - 1;
        const float4 r = S.rim[j * 32 + f];
        const float E = dec_edge(r.x, r.y, r.z, r.w, pxc, pyc);
        const bool fl = (flip >> j) & 1u;
        const bool in = E == 0.0f ? (fl ? edge_tie(-r.x, -r.y) : edge_tie(r.x, r.y)) : (E > 0.0f) != fl;
        hits |= (uint32_t)in << j;
    }
    return hits;
}

template <int TILE, int KT>
__device__ __forceinline__ void count_item(const RastArgs &a, char *smem, uint32_t item) {
    const int K = KT > 0 ? KT : a.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint4 it = a.items[item];
    const int view = view_of_tile(a.vt, it.x);
    const ViewDev &vw = a.vt.v[view];
    const int W = vw.cam.width, H = vw.cam.height;
    const float4 *dec = a.dec + (size_t)view * (size_t)a.V;
    const int tile = (int)(it.x - vw.tile_base), tiles_x = (int)vw.tiles_x;
    const CountMem S = count_mem<TILE>(smem + (size_t)warp * count_warp_bytes<TILE>(K), K);
    const int tx0 = (tile % tiles_x) * TILE, ty0 = (tile / tiles_x) * TILE;
    const int tx1 = min(tx0 + TILE, W) - 1, ty1 = min(ty0 + TILE, H) - 1;
    for (int i = lane; i < TILE * TILE; i += 32) S.cnt[i] = 0;
    const uint32_t lt = (1u << lane) - 1u, le = 0xffffffffu >> (31 - lane);
    for (uint32_t cb = it.y; cb < it.z; cb += 32) {
        const bool mine = cb + lane < it.z;
        uint32_t geo = 0;
        __syncwarp();   // the previous pairs are done with the stage
        if (mine) {
            const uint32_t fan = __ldg(a.list + cb + lane);
            const float4 *dv = dec + (size_t)fan * (K + 1);   // the binning pass's decide_vertex, bit for bit
            const float4 c = __ldg(dv), b0 = __ldg(dv + 1);
            const int ox = (int)c.w, oy = (int)b0.w;
            const uint32_t drawn = a.face_mask ? __ldg(a.face_mask + fan) : 0xffffffffu;
            float mnx = c.x, mxx = c.x, mny = c.y, mxy = c.y;
            uint32_t flags = 0, any = 0;
            float4 b = b0;
#pragma unroll(KT > 0 ? KT : 1)
            for (int j = 0; j < K; ++j) {
                const bool wrap = j + 1 == K;
                const float4 n = wrap ? b0 : __ldg(dv + 2 + j);
                // (binning marks invalid vertices with Z = -1)
                const bool valid = c.z > 0.0f && b.z > 0.0f && n.z > 0.0f && ((drawn >> j) & 1u);
                if (valid) {   // bounds over the vertices of valid triangles
                    any = 1;
                    mnx = fminf(mnx, fminf(b.x, n.x)); mxx = fmaxf(mxx, fmaxf(b.x, n.x));
                    mny = fminf(mny, fminf(b.y, n.y)); mxy = fmaxf(mxy, fmaxf(b.y, n.y));
                }
                S.sd[j * 32 + lane] = make_float2(__fsub_rn(b.x, c.x), __fsub_rn(b.y, c.y));
                S.rim[j * 32 + lane] = wrap ? make_float4(__fsub_rn(b.x, n.x), __fsub_rn(b.y, n.y), n.x, n.y)
                                            : make_float4(__fsub_rn(n.x, b.x), __fsub_rn(n.y, b.y), b.x, b.y);
                const float ar = dec_area2(c.x, c.y, b.x, b.y, n.x, n.y);
                if (valid && ar != 0.0f) flags |= 1u << j;
                if (ar < 0.0f) flags |= 1u << (16 + j);
                b = n;
            }
            S.flags[lane] = flags;
            S.c[lane] = make_float4((float)(tx0 - ox) + 0.5f, (float)(ty0 - oy) + 0.5f, c.x, c.y);
            const FanRect r = rect_from_bounds_rel(mnx, mxx, mny, mxy, ox, oy, W, H);
            const int rx0 = max(r.i0, tx0), rx1 = min(r.i1, tx1), ry0 = max(r.j0, ty0), ry1 = min(r.j1, ty1);
            if (any && (flags & 0xffffu) && !r.empty && rx0 <= rx1 && ry0 <= ry1)
                geo = pair_geo(rx0 - tx0, ry0 - ty0, rx1 - rx0 + 1, ry1 - ry0 + 1);
        }
        const uint32_t w = ((geo >> 12) & 63u) + 1u, h = ((geo >> 18) & 63u) + 1u;
        const bool in = geo != 0u;
        // runs in the low half, tests in the high half: at most 32 x 32 x 32 of each
        const uint32_t own = in ? h * ((w + 1u) / 2u) | (h * w) << 16 : 0u;
        uint32_t sum = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += y;
        }
        const uint32_t all = __shfl_sync(0xffffffffu, sum, 31), total = all & 0xffffu;
        const uint32_t excl = (sum - own) & 0xffffu, excl_t = (sum - own) >> 16;
        // The coverage mask of every test is stored (one range per 32 pairs, reserved with one
        // atomic) with each pair's first index; the fill pass reads them instead of testing again.
        // Both walk a fan's rectangle in the same order.  Up to kMaskRegions cursors, the item
        // picking one by its index, so that the reservations do not queue on one address.
        uint32_t mbase = ~0u;
        if (lane == 0 && total > 0) {
            const uint32_t reg = item % a.mask_regions;
            const uint32_t rsz = (uint32_t)(a.mask_cap / a.mask_regions);
            const unsigned long long b = atomicAdd(a.mask_cursor + reg, (unsigned long long)(all >> 16));
            if (b + (all >> 16) <= rsz) mbase = reg * rsz + (uint32_t)b;
        }
        mbase = __shfl_sync(0xffffffffu, mbase, 0);
        const uint32_t live = __ballot_sync(0xffffffffu, in);   // pairs with tests, in order
        if (in) S.info[__popc(live & lt)] = make_uint4(excl, excl_t, geo, (uint32_t)lane);
        __syncwarp();
        uint32_t fan_hit = 0;   // bit f set when the pair of lane f covers some pixel centre
        for (uint32_t base = 0; base < total; base += 32) {
            // the pair of each run: the pairs' runs start one after another, so a run's pair is the
            // last one that starts at or before it
            const int before = __popc(__ballot_sync(0xffffffffu, in && excl < base));
            const uint32_t here = in && excl >= base && excl < base + 32 ? 1u << (excl - base) : 0u;
            const uint32_t starts = __reduce_or_sync(0xffffffffu, here);
            const uint4 inf = S.info[before + __popc(starts & le) - 1];
            const uint32_t idx = base + lane;
            uint32_t hits0 = 0, hits1 = 0;
            if (idx < total) {
                const int f = (int)inf.w;
                const uint32_t local = idx - inf.x, fw = ((inf.z >> 12) & 63u) + 1u, runs = (fw + 1u) / 2u;
                // (local + 0.5) / runs is at least 1/(2 runs) away from an integer: exact row
                const uint32_t yy = (uint32_t)__fdividef((float)local + 0.5f, (float)runs);
                const uint32_t xx = 2u * (local - yy * runs);
                const uint32_t x = (inf.z & 63u) + xx, y = ((inf.z >> 6) & 63u) + yy;
                const bool two = xx + 1u < fw;
                // decisions in the fan's relative frame (its origin is an integer: the sums are exact)
                const float4 c = S.c[f];
                const float px0 = c.x + (float)x, px1 = px0 + 1.0f, py = c.y + (float)y;
                const float q0 = __fsub_rn(px0, c.z), q1 = __fsub_rn(px1, c.z), qy = __fsub_rn(py, c.w);
                uint32_t N0 = 0, N1 = 0;
                float least0 = 3.0e38f, least1 = 3.0e38f;
#pragma unroll(KT > 0 ? KT : 1)
                for (int i = K - 1; i >= 0; --i) {   // (descending, so that spoke i lands in bit i)
                    const float2 d = S.sd[i * 32 + f];
                    const float t = __fmul_rn(d.x, qy);
                    const float S0 = __fsub_rn(t, __fmul_rn(d.y, q0)), S1 = __fsub_rn(t, __fmul_rn(d.y, q1));
                    N0 = __funnelshift_l(__float_as_uint(S0), N0, 1);
                    N1 = __funnelshift_l(__float_as_uint(S1), N1, 1);
                    least0 = fminf(least0, fabsf(S0));
                    least1 = fminf(least1, fabsf(S1));
                }
                const uint32_t flags = S.flags[f];
                hits0 = cover_mask<KT>(S, K, f, flags, N0, least0 == 0.0f, px0, py, q0, qy);
                if (two) hits1 = cover_mask<KT>(S, K, f, flags, N1, least1 == 0.0f, px1, py, q1, qy);
                if (mbase != ~0u) {
                    uint16_t *m = a.masks + (mbase + inf.y + yy * fw + xx);
                    m[0] = (uint16_t)hits0;
                    if (two) m[1] = (uint16_t)hits1;
                }
                // the order of a pixel's slots does not matter
                uint32_t *cnt = S.cnt + (y * TILE + x);
                if (hits0) atomicAdd(cnt, (uint32_t)__popc(hits0));
                if (hits1) atomicAdd(cnt + 1, (uint32_t)__popc(hits1));
            }
            fan_hit |= __reduce_or_sync(0xffffffffu, hits0 | hits1 ? 1u << inf.w : 0u);
        }
        // each pair's first mask index, and its rectangle if it covers any pixel centre
        if (mine)
            a.pinfo[cb + lane] = make_uint2(mbase == ~0u ? ~0u : mbase + excl_t, ((fan_hit >> lane) & 1u) ? geo : 0u);
    }
    __syncwarp();
    uint32_t *icnt = a.icnt + (size_t)item * TILE * TILE;
    for (int i = lane; i < TILE * TILE; i += 32) {
        const uint32_t c = S.cnt[i];   // (nonzero only inside the image)
        if (c)
            icnt[i] = atomicAdd(a.counts + vw.pix_base + (size_t)(ty0 + i / TILE) * W + (size_t)(tx0 + i % TILE), c);
    }
}

template <int TILE, int KT, bool STRIDED>
__global__ void __launch_bounds__(kRastWarps * 32) count_kernel(const __grid_constant__ RastArgs a) {
    extern __shared__ __align__(16) char smem[];
    const uint32_t n_items = a.st->n_items;
    uint32_t item = blockIdx.x * kRastWarps + threadIdx.x / 32;   // (whole warps: nothing synchronises the block)
    if (!STRIDED) {
        if (item < n_items) count_item<TILE, KT>(a, smem, item);
    } else {
        for (; item < n_items; item += gridDim.x * kRastWarps) {
            count_item<TILE, KT>(a, smem, item);
            __syncwarp();   // the stage is free again
        }
    }
}

template <int TILE, int KT>
cudaError_t launch_t(const RastArgs &ra, int64_t max_items, int K, cudaStream_t st) {
    const size_t smem = kRastWarps * count_warp_bytes<TILE>(K);
    const int64_t blocks = (max_items + kRastWarps - 1) / kRastWarps;
    const bool strided = blocks > kItemBlocks;
    auto fn = strided ? count_kernel<TILE, KT, true> : count_kernel<TILE, KT, false>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    fn<<<(unsigned)(strided ? kStrideBlocks : blocks), kRastWarps * 32, smem, st>>>(ra);
    return cudaGetLastError();
}

template <int TILE>
cudaError_t launch_k(const RastArgs &ra, int64_t max_items, int K, cudaStream_t st) {
    if (K == 8) return launch_t<TILE, 8>(ra, max_items, K, st);
    if (K == 6) return launch_t<TILE, 6>(ra, max_items, K, st);
    return launch_t<TILE, 0>(ra, max_items, K, st);
}

RastArgs make_args(const RenderArgs &ra) {
    const RenderLayout &L = ra.L;
    RastArgs a;
    a.K = ra.K;
    a.vt = ra.vt;
    a.list = reinterpret_cast<const uint32_t *>(ra.ws + L.off_list);
    a.counts = reinterpret_cast<uint32_t *>(ra.ws + L.off_counts);
    a.items = reinterpret_cast<const uint4 *>(ra.ws + L.off_items);
    a.icnt = reinterpret_cast<uint32_t *>(ra.ws + L.off_icnt);
    a.st = reinterpret_cast<Status *>(ra.ws + L.off_status);
    a.dec = reinterpret_cast<const float4 *>(ra.ws + L.off_dec);
    a.V = L.V;
    a.face_mask = ra.prm.face_mask;
    a.pinfo = reinterpret_cast<uint2 *>(ra.ws + L.off_maskoff);
    a.masks = reinterpret_cast<uint16_t *>(ra.ws + L.off_masks);
    a.mask_cap = L.mask_cap;
    // regions of at least 2^19 masks: 32 pairs of a whole tile take 2^15, and few regions fill evenly
    a.mask_regions = (uint32_t)std::min<int64_t>(kMaskRegions, std::max<int64_t>(1, L.mask_cap >> 19));
    a.mask_cursor = reinterpret_cast<unsigned long long *>(ra.ws + L.off_mask_cursor);
    return a;
}

}  // namespace

cudaError_t launch_count(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    if (L.n_tiles == 0) return cudaSuccess;
    const RastArgs a = make_args(ra);
    const cudaError_t e = L.tile == 8    ? launch_k<8>(a, L.max_items, ra.K, st)
                          : L.tile == 32 ? launch_k<32>(a, L.max_items, ra.K, st)
                                         : launch_k<16>(a, L.max_items, ra.K, st);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

}  // namespace ms
