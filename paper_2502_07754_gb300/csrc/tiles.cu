// Tile lists of the rasteriser and the record ranges of its pixels.
//
// Binning leaves (tile, fan) pairs with each pair's rank within its tile and every tile's pair
// count.  tile_scan_kernel turns the counts into list starts and cuts the lists into work items
// (one warp each in the count and fill passes); tile_scatter_kernel writes each fan to its
// place.  A list's order does not matter (the resolve sorts a pixel's fragments by their exact
// depths), so this counting sort by tile replaces a radix sort by (tile, depth): per pair 20 bytes
// written and read once each, instead of 8 read and 8 written per digit pass.
// 1M fans (1.34M pairs): 15 us against 146 us for depth range, histogram, four digit passes, ranges
// and items; 3M fans in 16 views (42M pairs): 0.14 against 1.5 ms.
//
// After the count pass, pixel_alloc_kernel gives every pixel its range of the fragment buffer:
// spans of 1024 pixel slots in tile order (slot s = tile * TILE^2 + row * TILE + column within the
// tile) take their records together, so the records of one screen tile are contiguous: the
// passes that walk the records in order (the adjoint chain) then find the same fans again
// within a few hundred records, and the fill's writes for a tile stay in one region of the buffer.
// The same kernel lists the pixels for the resolve by class of fragment count (more than 32, 17
// to 32, 9 to 16, 1 to 8), in descending count within a span, and writes the background of
// pixels without fragments: one read of the counts, where a scan over the pixels (40 us at 1080p),
// a per-tile prefix over the items (99 us) and a global order by count (16 us) took 24 us here.
#include "raster_common.cuh"

namespace ms {

namespace {

// Exclusive scan over the tiles (decoupled look-back over virtual block ids, bounded waits) of
// (pairs, work items), packed in one word: pairs in the low 31 bits, items in the next 31.
constexpr int kTScanThreads = 256, kTScanItems = 2, kTScanTile = kTScanThreads * kTScanItems;
constexpr unsigned long long kFlagAgg = 1ull << 62, kFlagPre = 2ull << 62, kValMask = (1ull << 62) - 1;

// Fans per work item: 64 amortise an item's setup, but a scene whose lists give the chip too
// few warps that way takes smaller items, as far as the item capacity goes and not below 4 (1k fans
// at 128x128, forward and adjoint: 191 us with 8, 175 with 4, 177 with 2).
__device__ __forceinline__ uint32_t item_fans(unsigned long long pairs, unsigned long long cap) {
    uint32_t f = kItemFans;
    while (f > 4 && pairs < 8192ull * f && pairs * kItemFans <= cap * (f / 2)) f >>= 1;
    return f;
}

__global__ void __launch_bounds__(kTScanThreads) tile_scan_kernel(const uint32_t *__restrict__ cnt, int n_tiles,
                                                                  int nblocks, unsigned long long *state, Status *st,
                                                                  uint32_t *__restrict__ start,
                                                                  uint4 *__restrict__ items, int64_t max_items,
                                                                  unsigned long long frag_cap) {
    __shared__ int s_vid;
    __shared__ unsigned long long s_warp[kTScanThreads / 32], s_excl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_vid = (int)atomicAdd(&st->tscan_ticket, 1u);
    __syncthreads();
    const int vid = s_vid;
    const uint32_t F = item_fans(min(st->pairs, st->cap), st->cap);
    const int t0 = vid * kTScanTile + tid * kTScanItems;
    uint32_t c[kTScanItems];
    unsigned long long sum = 0;
#pragma unroll
    for (int i = 0; i < kTScanItems; ++i) {
        c[i] = t0 + i < n_tiles ? cnt[t0 + i] : 0u;
        sum += (unsigned long long)c[i] | (unsigned long long)((c[i] + F - 1) / F) << 31;
    }
    unsigned long long x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    unsigned long long before = 0, total = 0;
    for (int w = 0; w < kTScanThreads / 32; ++w) {
        if (w < warp) before += s_warp[w];
        total += s_warp[w];
    }
    if (tid == 0) {
        unsigned long long excl = 0;
        if (vid > 0) {
            st_release_u64(&state[vid], kFlagAgg | total);
            int j = vid - 1;
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
        }
        st_release_u64(&state[vid], kFlagPre | ((excl + total) & kValMask));
        s_excl = excl;
        if (vid == nblocks - 1) {
            const unsigned long long ni = (excl + total) >> 31;
            st->items_total = ni;
            st->n_items = (unsigned)(ni < (unsigned long long)max_items ? ni : (unsigned long long)max_items);
            st->frag_cap = frag_cap;
        }
    }
    __syncthreads();
    unsigned long long run = s_excl + before + x - sum;
#pragma unroll
    for (int i = 0; i < kTScanItems; ++i) {
        if (t0 + i >= n_tiles) break;
        const uint32_t s0 = (uint32_t)(run & 0x7fffffffull), n = (c[i] + F - 1) / F;
        const int64_t i0 = (int64_t)(run >> 31);
        start[t0 + i] = s0;
        for (uint32_t k = 0; k < n; ++k)
            if (i0 + k < max_items)
                items[i0 + k] = make_uint4((uint32_t)(t0 + i), s0 + k * F, s0 + min(c[i], (k + 1) * F), k);
        run += (unsigned long long)c[i] | (unsigned long long)n << 31;
    }
}

__global__ void __launch_bounds__(256) tile_scatter_kernel(const uint2 *__restrict__ pairs,
                                                           const uint32_t *__restrict__ ranks, const Status *st,
                                                           int64_t cap, const uint32_t *__restrict__ start,
                                                           uint32_t *__restrict__ list) {
    const int64_t n = min64((int64_t)st->pairs, cap);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {   // four pairs in flight per thread
        uint2 p[4];
        uint32_t r[4], s[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            p[u] = __ldg(pairs + i + u * stride);
            r[u] = __ldg(ranks + i + u * stride);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) s[u] = __ldg(start + p[u].x);
#pragma unroll
        for (int u = 0; u < 4; ++u) list[s[u] + r[u]] = p[u].y;
    }
    for (; i < n; i += stride) {
        const uint2 p = __ldg(pairs + i);
        list[__ldg(start + p.x) + __ldg(ranks + i)] = p.y;
    }
}

constexpr int kAllocThreads = 256, kAllocSlots = 4, kAllocSpan = kAllocThreads * kAllocSlots;

struct AllocArgs {
    int64_t npx, n_slots, order_b, frag_cap;
    int tile_shift;
    const uint32_t *counts;
    uint32_t *offsets;
    uint2 *list_a;              // pixel lists: see ResolveArgs (resolve.cu)
    uint32_t *list_b;
    float *tfinal;
    Status *st;
    const unsigned long long *tests;   // [kMaskRegions] tests of the count pass, in parts
    float bg0, bg1, bg2;
    ViewTable vt;
};

__global__ void __launch_bounds__(kAllocThreads) pixel_alloc_kernel(const __grid_constant__ AllocArgs a) {
    __shared__ uint32_t s_cnt[kCountBuckets], s_at[kCountBuckets], s_warp[kAllocThreads / 32], s_class[4], s_base[4];
    __shared__ unsigned long long s_sum[kAllocThreads / 32], s_first;
    static_assert(kAllocThreads == kCountBuckets, "one thread per bucket");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    s_cnt[tid] = 0;
    if (tid < 4) s_class[tid] = 0;
    if (blockIdx.x == 0) {
        static_assert(kMaskRegions <= kAllocThreads, "one thread per part");
        unsigned long long t = tid < kMaskRegions ? a.tests[tid] : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0 && t) atomicAdd(&a.st->rect_tests, t);
    }
    // this thread's four slots: neighbours in a row of one tile
    const int64_t s0 = (int64_t)blockIdx.x * kAllocSpan + tid * kAllocSlots;
    uint32_t n[kAllocSlots] = {0, 0, 0, 0};
    int64_t pix = 0, lpix = 0;
    int in = 0, view = 0;   // slots inside the image
    if (s0 < a.n_slots) {
        const uint32_t t = (uint32_t)(s0 >> (2 * a.tile_shift));
        const int local = (int)(s0 & ((1 << (2 * a.tile_shift)) - 1));
        view = view_of_tile(a.vt, t);
        const ViewDev &vw = a.vt.v[view];
        const uint32_t lt = t - vw.tile_base, tiles_x = vw.tiles_x, ty = lt / tiles_x, tx = lt - ty * tiles_x;
        const int x = (int)(tx << a.tile_shift) + (local & ((1 << a.tile_shift) - 1));
        const int y = (int)(ty << a.tile_shift) + (local >> a.tile_shift);
        if (y < vw.cam.height) in = max(0, min(kAllocSlots, vw.cam.width - x));
        lpix = (int64_t)y * vw.cam.width + x;
        pix = (int64_t)vw.pix_base + lpix;
        for (int i = 0; i < in; ++i) n[i] = a.counts[pix + i];
    }
    // (64 bits: millions of fans over one span, counted without room for their records, pass 2^32 fragments)
    const unsigned long long sum = (unsigned long long)n[0] + n[1] + n[2] + n[3];
    unsigned long long x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_sum[warp] = x;
    __syncthreads();
    unsigned long long before = 0, total = 0;
    for (int w = 0; w < kAllocThreads / 32; ++w) {
        if (w < warp) before += s_sum[w];
        total += s_sum[w];
    }
    if (tid == 0) s_first = total ? atomicAdd(&a.st->frags, total) : 0ull;
    __syncthreads();
    unsigned long long run = s_first + before + x - sum;
    // rank of each pixel among the span's pixels of its count; a pixel whose records do not fit the buffer
    // (reported through the status block) is none of them, so the lists cannot overflow
    int bk[kAllocSlots];
    uint32_t rk[kAllocSlots];
    {
        unsigned long long end = run;
#pragma unroll
        for (int i = 0; i < kAllocSlots; ++i) {
            end += n[i];
            bk[i] = end <= (unsigned long long)a.frag_cap ? count_bucket(n[i]) : 0;
            rk[i] = bk[i] ? atomicAdd(&s_cnt[bk[i]], 1u) : 0u;
        }
    }
    __syncthreads();
    // descending prefix over the counts: thread t holds count 255 - t
    const int mb = kCountBuckets - 1 - tid;
    const uint32_t h = mb ? s_cnt[mb] : 0u;
    uint32_t px = h;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, px, o);
        if (lane >= o) px += y;
    }
    if (lane == 31) s_warp[warp] = px;
    const int cls = mb > 32 ? 0 : (mb > 16 ? 1 : (mb > 8 ? 2 : 3));
    if (h) atomicAdd(&s_class[cls], h);
    __syncthreads();
    for (int w = 0; w < warp; ++w) px += s_warp[w];
    if (tid < 4) s_base[tid] = s_class[tid] ? atomicAdd(&a.st->classes[tid], s_class[tid]) : 0u;
    // place within the class
    uint32_t skip = 0;
    for (int c = 0; c < cls; ++c) skip += s_class[c];
    s_at[mb] = px - h - skip;
    __syncthreads();
    const ViewDev &vw = a.vt.v[view];
    for (int i = 0; i < in; ++i) {
        // offsets beyond 2^32 are clamped; such a buffer overflows its capacity anyway
        const uint32_t off = (uint32_t)(run < 0xffffffffull ? run : 0xffffffffull);
        run += n[i];
        a.offsets[pix + i] = off;
        if (bk[i]) {
            const int c = bk[i] > 32 ? 0 : (bk[i] > 16 ? 1 : (bk[i] > 8 ? 2 : 3));
            const int64_t at = (int64_t)s_base[c] + s_at[bk[i]] + rk[i];
            const uint2 e = make_uint2((uint32_t)(pix + i), off);
            if (c == 0) a.list_b[a.order_b - 1 - at] = e.x;
            if (c == 1) a.list_b[at] = e.x;
            if (c == 2) a.list_a[a.npx - 1 - at] = e;
            if (c == 3) a.list_a[at] = e;
        } else {   // no fragments, or no room for them: the background
            reinterpret_cast<float4 *>(vw.out)[lpix + i] = make_float4(a.bg0, a.bg1, a.bg2, 0.0f);
            a.tfinal[pix + i] = 1.0f;
        }
    }
}

}  // namespace

int64_t tile_scan_blocks(int64_t n_tiles) { return (n_tiles + kTScanTile - 1) / kTScanTile; }

cudaError_t launch_tile_lists(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    char *ws = ra.ws;
    Status *status = reinterpret_cast<Status *>(ws + L.off_status);
    uint32_t *start = reinterpret_cast<uint32_t *>(ws + L.off_tile_start);
    tile_scan_kernel<<<(unsigned)L.tscan_blocks, kTScanThreads, 0, st>>>(
        reinterpret_cast<const uint32_t *>(ws + L.off_tile_cnt), L.n_tiles, (int)L.tscan_blocks,
        reinterpret_cast<unsigned long long *>(ws + L.off_tscan_state), status, start,
        reinterpret_cast<uint4 *>(ws + L.off_items), L.max_items, (unsigned long long)L.frag_cap);
    const unsigned grid = (unsigned)min64((L.cap + 255) / 256, 8 * 152);
    tile_scatter_kernel<<<grid, 256, 0, st>>>(reinterpret_cast<const uint2 *>(ws + L.off_pairs),
                                              reinterpret_cast<const uint32_t *>(ws + L.off_ranks), status, L.cap,
                                              start, reinterpret_cast<uint32_t *>(ws + L.off_list));
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) count_launches(2);
    return e;
}

cudaError_t launch_pixel_alloc(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    char *ws = ra.ws;
    AllocArgs a;
    a.npx = L.npx;
    a.tile_shift = 0;
    while ((1 << a.tile_shift) < L.tile) ++a.tile_shift;
    a.n_slots = (int64_t)L.n_tiles << (2 * a.tile_shift);
    a.order_b = L.order_b;
    a.frag_cap = L.frag_cap;
    a.counts = reinterpret_cast<const uint32_t *>(ws + L.off_counts);
    a.offsets = reinterpret_cast<uint32_t *>(ws + L.off_offsets);
    a.list_a = reinterpret_cast<uint2 *>(ws + L.off_order_a);
    a.list_b = reinterpret_cast<uint32_t *>(ws + L.off_order_b);
    a.tfinal = reinterpret_cast<float *>(ws + L.off_tfinal);
    a.st = reinterpret_cast<Status *>(ws + L.off_status);
    a.tests = reinterpret_cast<const unsigned long long *>(ws + L.off_mask_cursor);
    a.bg0 = ra.prm.bg[0];
    a.bg1 = ra.prm.bg[1];
    a.bg2 = ra.prm.bg[2];
    a.vt = ra.vt;
    pixel_alloc_kernel<<<(unsigned)((a.n_slots + kAllocSpan - 1) / kAllocSpan), kAllocThreads, 0, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) count_launches(1);
    return e;
}

}  // namespace ms
