// Tile rasterisation into a per-pixel fragment buffer (A-buffer) in HBM: the count pass.
//
// Every tile's fan list is cut into work items of at most kItemFans fans (tiles.cu); one warp
// rasterises one item, so a hot tile with thousands of fans spreads over many warps instead of
// serialising on one.  A warp stages the decisions of a chunk of the item's fans in its own
// shared memory (32 / chunk lanes per fan, sharing its vertices and triangles); the staged
// fans' pixel rectangles inside the tile form one index space of (fan, pixel) tests, a lane
// each, which the binary32 decision formulas answer for the fan's K triangles.  No block
// barriers are used.
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
    uint32_t *mask_cursor;     // [mask_regions] fill levels of the mask regions (zeroed per render)
};

constexpr int kRastWarps = 2;   // warps (work items) per block: items differ widely in cost

template <int TILE, int STG>
__host__ __device__ __forceinline__ size_t warp_smem_bytes(int K) {
    return (size_t)(TILE * TILE + 32) * 4 + stage_bytes(STG, K);
}

template <int TILE, int STG, int KT>
__global__ void __launch_bounds__(kRastWarps * 32) count_kernel(const __grid_constant__ RastArgs a) {
    extern __shared__ __align__(16) char smem[];
    const int K = KT > 0 ? KT : a.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t item = blockIdx.x * kRastWarps + warp;
    if (item >= a.st->n_items) return;   // whole warp; nothing below synchronises the block
    const uint4 it = a.items[item];
    const int view = view_of_tile(a.vt, it.x);
    const ViewDev &vw = a.vt.v[view];
    SceneDev sc;
    sc.W = vw.cam.width;
    sc.H = vw.cam.height;
    sc.dec = a.dec + (size_t)view * (size_t)a.V;
    sc.face_mask = a.face_mask;
    const int tile = (int)(it.x - vw.tile_base);
    const int tiles_x = (int)vw.tiles_x;
    char *mine = smem + (size_t)warp * warp_smem_bytes<TILE, STG>(K);
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(mine);   // [TILE*TILE] fragments so far
    uint32_t *s_map = s_cnt + TILE * TILE;                    // [32] staged fans that have tests
    const Stage S = stage_ptrs(mine + (size_t)(TILE * TILE + 32) * 4, STG, K);
    const int tx0 = (tile % tiles_x) * TILE, ty0 = (tile / tiles_x) * TILE;
    const int tx1 = min(tx0 + TILE, sc.W) - 1, ty1 = min(ty0 + TILE, sc.H) - 1;
    for (int i = lane; i < TILE * TILE; i += 32) s_cnt[i] = 0;
    uint32_t c_rect = 0, c_frag = 0;
    __syncwarp();
    for (uint32_t cb = it.y; cb < it.z; cb += STG) {
        const int cnt = (int)min((uint32_t)STG, it.z - cb);
        {
            constexpr int LPF = 32 / STG;   // lanes staging one fan
            const int slot = lane / LPF;
            uint32_t fan = 0;
            if (slot < cnt) fan = __ldg(a.list + cb + slot);
            stage_fans<LPF>(sc, S, K, lane, slot < cnt, fan);
        }
        __syncwarp();
        // The staged fans' rectangles (clipped to the tile) form one packed (fan, pixel)
        // index space, fan-major, so every lane tests a pixel even when fans are tiny.
        int my_n = 0;
        uint32_t my_geo = 0;
        if (lane < cnt) {
            const int4 r = S.rect[lane];
            const int rx0 = max(r.x, tx0), rx1 = min(r.y, tx1), ry0 = max(r.z, ty0), ry1 = min(r.w, ty1);
            if (S.flags[lane] != 0 && rx0 <= rx1 && ry0 <= ry1)
                my_geo = pair_geo(rx0 - tx0, ry0 - ty0, rx1 - rx0 + 1, ry1 - ry0 + 1);
        }
        if (my_geo) my_n = (int)((((my_geo >> 12) & 63u) + 1u) * (((my_geo >> 18) & 63u) + 1u));
        int incl = my_n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int excl = incl - my_n;
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        // The coverage mask of every test of the chunk is stored (one range per chunk, reserved
        // with one atomic) with each pair's first index; the fill pass reads them instead of
        // testing again.  Both walk a fan's rectangle in the same order.
        uint32_t mbase = ~0u;
        {
            // up to kMaskRegions cursors, the item picking one by its index, so that the
            // reservations of millions of chunks do not queue on one address
            if (lane == 0 && total > 0) {
                const uint32_t reg = item % a.mask_regions;
                const uint32_t rsz = (uint32_t)(a.mask_cap / a.mask_regions);
                const uint32_t b = atomicAdd(a.mask_cursor + reg, (uint32_t)total);
                if ((uint64_t)b + (uint64_t)total <= (uint64_t)rsz) mbase = reg * rsz + b;
            }
            mbase = __shfl_sync(0xffffffffu, mbase, 0);
        }
        const uint32_t live = __ballot_sync(0xffffffffu, my_n != 0);   // staged fans with tests, in order
        if (my_n) s_map[__popc(live & ((1u << lane) - 1u))] = (uint32_t)lane;
        __syncwarp();
        uint32_t fan_hit = 0;   // bit f set when staged fan f covers some pixel centre
        for (int base = 0; base < total; base += 32) {
            const int idx = base + lane;
            // the fan of each index: the fans with tests start one after another, so an index's
            // fan is the last one that starts at or before it
            const int before = __popc(__ballot_sync(0xffffffffu, my_n != 0 && excl < base));
            const uint32_t here = my_n != 0 && excl >= base && excl < base + 32 ? 1u << (excl - base) : 0u;
            const uint32_t starts = __reduce_or_sync(0xffffffffu, here);
            const int f = (int)s_map[before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1];
            const int fexcl = __shfl_sync(0xffffffffu, excl, f);
            const uint32_t fgeo = __shfl_sync(0xffffffffu, my_geo, f);
            uint32_t hits = 0;
            if (idx < total) {
                ++c_rect;
                const int local = idx - fexcl, w = (int)((fgeo >> 12) & 63u) + 1;
                // (local + 0.5) / w is at least 1/(2w) away from an integer: exact row
                const int yy = (int)__fdividef((float)local + 0.5f, (float)w);
                const int x = (int)(fgeo & 63u) + (local - yy * w), y = (int)((fgeo >> 6) & 63u) + yy;
                // decisions in the fan's relative frame (the origin is an integer)
                hits = cover_mask<KT>(S, STG, K, f, S.flags[f], (float)(tx0 + x - (int)S.ox[f]) + 0.5f,
                                      (float)(ty0 + y - (int)S.oy[f]) + 0.5f);
                if (mbase != ~0u) a.masks[mbase + (uint32_t)idx] = (uint16_t)hits;
                // the order of a pixel's slots does not matter yet
                if (hits) atomicAdd(&s_cnt[y * TILE + x], (uint32_t)__popc(hits));
            }
            fan_hit |= __reduce_or_sync(0xffffffffu, hits ? 1u << f : 0u);
            c_frag += __popc(hits);
        }
        // each pair's first mask index, and its rectangle if it covers any pixel centre
        if (lane < cnt)
            a.pinfo[cb + lane] = make_uint2(mbase == ~0u ? ~0u : mbase + (uint32_t)excl,
                                            ((fan_hit >> lane) & 1u) ? my_geo : 0u);
        __syncwarp();
    }
    uint32_t *icnt = a.icnt + (size_t)item * TILE * TILE;
    for (int i = lane; i < TILE * TILE; i += 32) {
        const uint32_t c = s_cnt[i];   // (nonzero only inside the image)
        if (c)
            icnt[i] = atomicAdd(a.counts + vw.pix_base + (size_t)(ty0 + i / TILE) * sc.W + (size_t)(tx0 + i % TILE), c);
    }
    const unsigned r0 = __reduce_add_sync(0xffffffffu, c_rect);
    const unsigned r1 = __reduce_add_sync(0xffffffffu, c_frag);
    if (lane == 0) {
        atomicAdd(&a.st->rect_tests, (unsigned long long)r0);
        atomicAdd(&a.st->fragments, (unsigned long long)r1);
    }
}

template <int TILE, int KT>
cudaError_t launch_t(const RastArgs &ra, int64_t max_items, int K, cudaStream_t st) {
    // fans staged per chunk: small enough that the shared-memory stage of a warp lets
    // many warps share an SM, large enough to keep the packed (fan, pixel) batches full
    constexpr int STG = 16;
    const size_t smem = kRastWarps * warp_smem_bytes<TILE, STG>(K);
    auto fn = count_kernel<TILE, STG, KT>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    fn<<<(unsigned)((max_items + kRastWarps - 1) / kRastWarps), kRastWarps * 32, smem, st>>>(ra);
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
    // regions of at least 2^16 masks, so that a small image's chunks (up to 16 fans of a whole
    // tile) fit one
    a.mask_regions = (uint32_t)std::min<int64_t>(kMaskRegions, std::max<int64_t>(1, L.mask_cap >> 16));
    a.mask_cursor = reinterpret_cast<uint32_t *>(ra.ws + L.off_mask_cursor);
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
