// Tile rasterisation into a per-pixel fragment buffer (A-buffer) in HBM.
//
// Every tile's fan list (sorted by the fans' depth bounds) is cut into work items of
// at most kItemFans fans; one warp rasterises one item, so a hot tile with thousands
// of fans spreads over many warps instead of serialising on one.  A warp projects
// a chunk of the item's fans into its own shared-memory stage (32 / chunk lanes per fan,
// sharing its vertices and triangles), then walks them in list order: for each fan its lanes enumerate exactly the pixels
// of the fan's pixel rectangle inside the tile and test the fan's K triangles at each
// with the binary32 decision formulas.  No block barriers are used.
//
// Count pass: per (item, pixel) fragment counts, the coverage mask of every (fan, pixel)
// test, and per pair its first mask index and its pixel rectangle within the tile (zero
// when the pair covers no pixel centre, so the fill skips it).  A
// per-tile prefix over the tile's items turns the counts into each item's starting slot
// within the pixel and gives the pixel totals; an exclusive scan over pixels gives record
// offsets.  The fill pass (fill.cu) walks the same items with the stored masks and rectangles
// and writes the records.
#include <algorithm>

#include "raster_common.cuh"

namespace ms {

namespace {

struct RastArgs {
    int K, fan_bits;
    ViewTable vt;
    const unsigned long long *keys;   // sorted elements tile | depth bound | fan id
    const uint4 *items;        // (tile, start, end, index within tile)
    uint32_t *icnt;            // [item][tile pixels]: counts, then in-pixel starting slots
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
    uint32_t *icnt = a.icnt + (size_t)item * TILE * TILE;
    for (int i = lane; i < TILE * TILE; i += 32) s_cnt[i] = 0;
    uint32_t c_rect = 0, c_frag = 0;
    __syncwarp();
    for (uint32_t cb = it.y; cb < it.z; cb += STG) {
        const int cnt = (int)min((uint32_t)STG, it.z - cb);
        {
            constexpr int LPF = 32 / STG;   // lanes staging one fan
            const int slot = lane / LPF;
            uint32_t fan = 0;
            if (slot < cnt) fan = (uint32_t)(__ldg(a.keys + cb + slot) & ((1ull << a.fan_bits) - 1ull));
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
    for (int i = lane; i < TILE * TILE; i += 32) icnt[i] = s_cnt[i];
    const unsigned r0 = __reduce_add_sync(0xffffffffu, c_rect);
    const unsigned r1 = __reduce_add_sync(0xffffffffu, c_frag);
    if (lane == 0) {
        atomicAdd(&a.st->rect_tests, (unsigned long long)r0);
        atomicAdd(&a.st->fragments, (unsigned long long)r1);
    }
}

// Exclusive scan of u32 counts into u32 offsets (decoupled look-back over virtual block
// ids, bounded waits); the grand total goes to *total_out.
//
// With SLOTS the scan runs over the pixels in tile order (slot s = tile * TILE^2 + row *
// TILE + column within the tile; slots outside the image count 0 and get no offset), so the
// fragment records of one screen tile are contiguous: the passes that walk the records in
// order (the adjoint chain) then find the same fans again within a few hundred records,
// and the fill's writes for a tile stay in one region of the buffer.
constexpr int kScanThreads = 256, kScanItems = 8, kScanTile = kScanThreads * kScanItems;
constexpr unsigned long long kFlagAgg = 1ull << 62, kFlagPre = 2ull << 62, kValMask = (1ull << 62) - 1;

// Pixel index of slot s (tile-ordered pixels), or -1 for a slot outside its view's image.
__device__ __forceinline__ int64_t slot_pixel(const ViewTable &vt, int tile_shift, int64_t s) {
    const uint32_t t = (uint32_t)(s >> (2 * tile_shift));
    const int local = (int)(s & ((1 << (2 * tile_shift)) - 1));
    const ViewDev &vw = vt.v[view_of_tile(vt, t)];
    const int lt = (int)(t - vw.tile_base), tiles_x = (int)vw.tiles_x;
    const int x = ((lt % tiles_x) << tile_shift) + (local & ((1 << tile_shift) - 1));
    const int y = ((lt / tiles_x) << tile_shift) + (local >> tile_shift);
    if (x >= vw.cam.width || y >= vw.cam.height) return -1;
    return (int64_t)vw.pix_base + (int64_t)y * vw.cam.width + x;
}

template <bool SLOTS>
__global__ void __launch_bounds__(kScanThreads) scan_u32_kernel(const uint32_t *__restrict__ counts,
                                                                uint32_t *__restrict__ offsets, int64_t n,
                                                                int64_t nblocks, unsigned long long *state,
                                                                unsigned *ticket, unsigned long long *total_out,
                                                                Status *st, const __grid_constant__ ViewTable vt,
                                                                int tile_shift) {
    __shared__ int s_vid;
    __shared__ uint32_t s_warp[kScanThreads / 32];
    __shared__ unsigned long long s_excl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_vid = (int)atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t vid = s_vid;
    const int64_t base = vid * kScanTile + (int64_t)tid * kScanItems;
    uint32_t v[kScanItems];
    int64_t pi[kScanItems];
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        pi[i] = base + i < n ? (SLOTS ? slot_pixel(vt, tile_shift, base + i) : base + i) : -1;
        v[i] = pi[i] >= 0 ? counts[pi[i]] : 0u;
        sum += v[i];
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t t = lane < kScanThreads / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < kScanThreads / 32) s_warp[lane] = t;
    }
    __syncthreads();
    const uint32_t total = s_warp[kScanThreads / 32 - 1];
    const uint32_t mine = x - sum + (warp > 0 ? s_warp[warp - 1] : 0);
    if (tid == 0) {
        unsigned long long excl = 0;
        if (vid == 0) {
            st_release_u64(&state[0], kFlagPre | (unsigned long long)total);
        } else {
            st_release_u64(&state[vid], kFlagAgg | (unsigned long long)total);
            int64_t j = vid - 1;
            uint32_t spins = 0;
            while (j >= 0) {
                const unsigned long long s = ld_acquire_u64(&state[j]);
                const unsigned long long flag = s & ~kValMask;
                if (flag == 0) {
                    if (++spins > kSpinLimit) {
                        atomicAdd(&st->timeouts, 1u);
                        break;
                    }
                    continue;
                }
                excl += s & kValMask;
                if (flag == kFlagPre) break;
                --j;
            }
            st_release_u64(&state[vid], kFlagPre | (excl + total));
        }
        s_excl = excl;
        if (vid == nblocks - 1) *total_out = excl + total;
    }
    __syncthreads();
    unsigned long long run = s_excl + mine;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        // offsets beyond 2^32 are clamped; such a buffer overflows its capacity anyway
        if (pi[i] >= 0) offsets[pi[i]] = (uint32_t)(run < 0xffffffffull ? run : 0xffffffffull);
        run += v[i];
    }
}

__global__ void tile_item_count_kernel(const uint2 *__restrict__ ranges, int n_tiles, uint32_t *__restrict__ nitems) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_tiles) {
        const uint32_t len = ranges[t].y - ranges[t].x;
        nitems[t] = (len + kItemFans - 1) / kItemFans;
    }
}

__global__ void tile_item_emit_kernel(const uint2 *__restrict__ ranges, int n_tiles, const uint32_t *__restrict__ nitems,
                                      const uint32_t *__restrict__ ibase, uint4 *__restrict__ items, int64_t max_items,
                                      Status *st, unsigned long long frag_cap) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) {
        const unsigned long long ni = st->items_total;
        st->n_items = (unsigned)(ni < (unsigned long long)max_items ? ni : (unsigned long long)max_items);
        st->frag_cap = frag_cap;
    }
    if (t >= n_tiles) return;
    const uint2 r = ranges[t];
    const uint32_t n = nitems[t], b = ibase[t];
    for (uint32_t k = 0; k < n; ++k)
        if (b + k < (uint64_t)max_items)
            items[b + k] = make_uint4((uint32_t)t, r.x + k * kItemFans, min(r.y, r.x + (k + 1) * kItemFans), k);
}

// Per tile: exclusive prefix of the (item, pixel) counts over the tile's items, the
// pixel totals, and their histogram by count_bucket (for the resolve's pixel order).  One block per tile, one thread per pixel; loads are issued four items
// at a time so a tile with many items is not latency-bound.
template <int TILE>
__global__ void __launch_bounds__(TILE *TILE) item_prefix_kernel(const uint32_t *__restrict__ nitems,
                                                                 const uint32_t *__restrict__ ibase,
                                                                 const __grid_constant__ ViewTable vt,
                                                                 uint32_t *__restrict__ icnt,
                                                                 uint32_t *__restrict__ counts,
                                                                 uint32_t *__restrict__ hist) {
    __shared__ uint32_t s_hist[kCountBuckets];
    const int t = blockIdx.x, i = threadIdx.x;
    for (int b = i; b < kCountBuckets; b += TILE * TILE) s_hist[b] = 0;
    const uint32_t n = nitems[t], b = ibase[t];
    uint32_t *c = icnt + (size_t)b * TILE * TILE + i;
    uint32_t run = 0;
    uint32_t k = 0;
    for (; k + 4 <= n; k += 4) {
        const uint32_t v0 = c[(size_t)k * TILE * TILE], v1 = c[(size_t)(k + 1) * TILE * TILE];
        const uint32_t v2 = c[(size_t)(k + 2) * TILE * TILE], v3 = c[(size_t)(k + 3) * TILE * TILE];
        c[(size_t)k * TILE * TILE] = run;
        c[(size_t)(k + 1) * TILE * TILE] = run + v0;
        c[(size_t)(k + 2) * TILE * TILE] = run + v0 + v1;
        c[(size_t)(k + 3) * TILE * TILE] = run + v0 + v1 + v2;
        run += v0 + v1 + v2 + v3;
    }
    for (; k < n; ++k) {
        const uint32_t v = c[(size_t)k * TILE * TILE];
        c[(size_t)k * TILE * TILE] = run;
        run += v;
    }
    const ViewDev &vw = vt.v[view_of_tile(vt, (uint32_t)t)];
    const int lt = t - (int)vw.tile_base, tiles_x = (int)vw.tiles_x;
    const int x = (lt % tiles_x) * TILE + (i % TILE), y = (lt / tiles_x) * TILE + (i / TILE);
    __syncthreads();
    if (x < vw.cam.width && y < vw.cam.height) {
        counts[vw.pix_base + (size_t)y * vw.cam.width + x] = run;
        atomicAdd(&s_hist[count_bucket(run)], 1u);
    }
    __syncthreads();
    for (int b = i; b < kCountBuckets; b += TILE * TILE)
        if (s_hist[b]) atomicAdd(&hist[b], s_hist[b]);
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

cudaError_t launch_count(const RastArgs &ra, const RenderLayout &L, int K, cudaStream_t st) {
    if (L.tile == 8) return launch_k<8>(ra, L.max_items, K, st);
    if (L.tile == 32) return launch_k<32>(ra, L.max_items, K, st);
    return launch_k<16>(ra, L.max_items, K, st);
}

RastArgs make_args(const RenderArgs &ra) {
    const RenderLayout &L = ra.L;
    RastArgs a;
    a.K = ra.K;
    a.vt = ra.vt;
    a.fan_bits = L.fan_bits;
    a.keys = reinterpret_cast<const unsigned long long *>(ra.ws + (L.passes & 1 ? L.off_keys1 : L.off_keys0));
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

cudaError_t launch_raster_count(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    char *ws = ra.ws;
    Status *status = reinterpret_cast<Status *>(ws + L.off_status);
    const RastArgs a = make_args(ra);
    const uint2 *ranges = reinterpret_cast<const uint2 *>(ws + L.off_ranges);
    uint32_t *nitems = reinterpret_cast<uint32_t *>(ws + L.off_tile_nitems);
    uint32_t *ibase = reinterpret_cast<uint32_t *>(ws + L.off_tile_ibase);
    const int tg = (L.n_tiles + 255) / 256;
    tile_item_count_kernel<<<tg, 256, 0, st>>>(ranges, L.n_tiles, nitems);
    scan_u32_kernel<false><<<(unsigned)L.tscan_blocks, kScanThreads, 0, st>>>(
        nitems, ibase, L.n_tiles, L.tscan_blocks, reinterpret_cast<unsigned long long *>(ws + L.off_tscan_state),
        &status->tscan_ticket, &status->items_total, status, ra.vt, 0);
    tile_item_emit_kernel<<<tg, 256, 0, st>>>(ranges, L.n_tiles, nitems, ibase,
                                              reinterpret_cast<uint4 *>(ws + L.off_items), L.max_items, status,
                                              (unsigned long long)L.frag_cap);
    cudaError_t e = ra.splat ? launch_splat_count(ra, st) : launch_count(a, L, ra.K, st);
    if (e != cudaSuccess) return e;
    uint32_t *cnts = reinterpret_cast<uint32_t *>(ws + L.off_counts);
    uint32_t *hist = reinterpret_cast<uint32_t *>(ws + L.off_pbucket);
    if (L.tile == 8)
        item_prefix_kernel<8><<<L.n_tiles, 64, 0, st>>>(nitems, ibase, ra.vt, a.icnt, cnts, hist);
    else if (L.tile == 32)
        item_prefix_kernel<32><<<L.n_tiles, 1024, 0, st>>>(nitems, ibase, ra.vt, a.icnt, cnts, hist);
    else
        item_prefix_kernel<16><<<L.n_tiles, 256, 0, st>>>(nitems, ibase, ra.vt, a.icnt, cnts, hist);
    int tile_shift = 0;
    while ((1 << tile_shift) < L.tile) ++tile_shift;
    const int64_t n = (int64_t)L.n_tiles << (2 * tile_shift);   // pixel slots in tile order
    scan_u32_kernel<true><<<(unsigned)L.scan_blocks, kScanThreads, 0, st>>>(
        reinterpret_cast<const uint32_t *>(ws + L.off_counts), reinterpret_cast<uint32_t *>(ws + L.off_offsets), n,
        L.scan_blocks, reinterpret_cast<unsigned long long *>(ws + L.off_scan_state), &status->scan_ticket,
        &status->frags, status, ra.vt, tile_shift);
    e = cudaGetLastError();
    if (e == cudaSuccess) count_launches(6);
    if (e == cudaSuccess) e = launch_pixel_order(ra, st);
    return e;
}

}  // namespace ms
