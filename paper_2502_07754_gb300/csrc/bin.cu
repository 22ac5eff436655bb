// Tile binning of fans: project, count overlapped tiles and emit one (tile, fan) pair per
// overlap with its rank within the tile -- one pass.  tiles.cu then puts the pairs in tile order.
//
// The binning unit is the fan (K triangles sharing the centre), not the single
// triangle: a fan is a few pixels wide, so one record per (tile, fan) instead of per
// (tile, triangle) cuts the pairs by about K.  A pair's rank is a counter of its tile; the lanes
// of a warp that hit one tile (neighbours in storage order mostly do) take their ranks with one
// atomic.
#include "dfloat2.cuh"
#include "fan_geom.cuh"
#include "ms_internal.h"

namespace ms {

namespace {

constexpr int kBinThreads = 256;

struct BinArgs {
    const float *xyz;
    int64_t n_fans;
    int K, tile_shift;
    int64_t cap, fan_blocks;
    unsigned n_tiles, sort_bits;
    Status *st;
    uint2 *pairs;              // (tile, fan)
    uint32_t *ranks;           // rank of each pair within its tile
    uint32_t *tile_cnt;        // pairs of each tile (zeroed per render)
    ViewTable vt;
    float4 *dec;               // [view][vertex] decided (xr, yr, Z or -1, origin), read by the raster passes
    int64_t V;
    const uint32_t *face_mask; // per fan, bit j = face j drawn; NULL = all
    bool splat;                // the soup holds polygons of splats (polygon_pad)
};

// How far, in pixels, the rounding of its binary32 vertices p (centre first, at depth zc) can draw the bounds of a
// splat's polygon inside the splat: a vertex moves by at most 2^-22 of the centre's coordinates (the
// additions) and 2^-20 of its offset from the centre (the rotated axes; no component of an offset exceeds the sum of
// those of the first and third boundary vertices, which lie on the axes), magnified by f + reach pixels at the least depth.
// 1e-3 px in a scene of a few units; 0.25 px at coordinates of 1000 seen from a unit away at f = 1000.
__device__ __forceinline__ float polygon_pad(const float *p, const CamDev &c, float zc, float reach) {
    float m = 0.0f, off = 0.0f, dz = 0.0f;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float o = fabsf(p[3 + r] - p[r]) + fabsf(p[9 + r] - p[r]);
        m = fmaxf(m, fabsf(p[r]));
        off = fmaxf(off, o);
        dz = fmaf(fabsf(c.R[6 + r]), o, dz);
    }
    const float f = fmaxf(fabsf(c.fx), fabsf(c.fy)) + reach;
    return fminf(__fdividef((0x1p-22f * m + 0x1p-20f * off) * f, fmaxf(zc - dz, c.znear)), 2.0f * kGuardPx);
}

// What bounds it: arithmetic (the double-float projection, two boundary vertices at a time: 83% of issue
// slots busy).  16 views of 3M fans, K = 6, forward and adjoint: 16.93 -> 16.62 ms against one vertex at a time in
// 48 registers; the pairs want 64 (four blocks an SM; with the 76 they would take, three, they gain nothing).
// Block = view * fan_blocks + fan block.  A block's pairs are contiguous and in fan order; the blocks' ranges come
// in the order in which they reserve them.
__global__ void __launch_bounds__(kBinThreads, 4) bin_kernel(const __grid_constant__ BinArgs a) {
    const float *__restrict__ xyz = a.xyz;
    const int64_t n_fans = a.n_fans;
    const int K = a.K, tile_shift = a.tile_shift;
    const int64_t cap = a.cap;
    Status *st = a.st;
    extern __shared__ float s_xyz[];   // kBinThreads * (K+1) * 3
    __shared__ uint32_t s_off[kBinThreads + 1];
    __shared__ uint32_t s_rect[kBinThreads][2];   // (tx0 | ty0 << 16), (w | h << 16)
    __shared__ uint32_t s_warp[kBinThreads / 32];
    __shared__ unsigned long long s_excl;
    __shared__ unsigned s_culled;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int KV = K + 1;
    if (tid == 0) s_culled = 0;
    __syncthreads();
    const int64_t vid = blockIdx.x;
    const int view = (int)(vid / a.fan_blocks);
    const int64_t f0 = (vid - (int64_t)view * a.fan_blocks) * kBinThreads;
    const int nloc = (int)min64(kBinThreads, n_fans - f0);
    const CamDev &cam = a.vt.v[view].cam;
    const unsigned tiles_x = a.vt.v[view].tiles_x, tile_base = a.vt.v[view].tile_base;

    // Coalesced staging of the block's vertices.
    {
        const float *src = xyz + f0 * KV * 3;
        const int n = nloc * KV * 3;
        if ((reinterpret_cast<uintptr_t>(src) & 15) == 0 && (n & 3) == 0) {
            const float4 *s4 = reinterpret_cast<const float4 *>(src);
            float4 *d4 = reinterpret_cast<float4 *>(s_xyz);
            for (int i = tid; i < n / 4; i += kBinThreads) d4[i] = __ldg(s4 + i);
        } else {
            for (int i = tid; i < n; i += kBinThreads) s_xyz[i] = __ldg(src + i);
        }
    }
    __syncthreads();

    uint32_t count = 0;
    if (tid < nloc) {
        const float *p = s_xyz + tid * KV * 3;
        const uint32_t all = (2u << K) - 1u;   // K+1 vertex bits
        uint32_t vmask = 0;
        float mnx = 3.0e38f, mxx = -3.0e38f, mny = 3.0e38f, mxy = -3.0e38f;
        float4 *dec = a.dec + (size_t)view * a.V + (size_t)(f0 + tid) * KV;
        // the fan's integer origin: the floor of its centre's exact screen position
        const DfVert c0 = df_project(cam, p[0], p[1], p[2]);
        const float ox = df_floor(c0.x), oy = df_floor(c0.y);
        // (xr, yr, Z or -1 if invalid, the origin's x / y in the first two vertices)
        auto take = [&](int k, const DVert &d, float w) {
            dec[k] = make_float4(d.xr, d.yr, d.valid ? d.Z : -1.0f, w);
            if (d.valid) vmask |= 1u << k;
            mnx = fminf(mnx, d.xs); mxx = fmaxf(mxx, d.xs);
            mny = fminf(mny, d.ys); mxy = fmaxf(mxy, d.ys);
        };
        take(0, decide_vertex(cam, c0, ox, oy), ox);
        const Cam2 cam_2 = cam2(cam);
        const F2 nox = f2_pack(-ox, -ox), noy = f2_pack(-oy, -oy);
        for (int k = 1; k <= K; k += 2) {   // two boundary vertices at a time
            const int kn = min(k + 1, K);
            DVert d, e;
            decide_vertex2(cam, cam_2, p + 3 * k, p + 3 * kn, nox, noy, d, e);
            take(k, d, k == 1 ? oy : 0.0f);
            if (k < K) take(k + 1, e, 0.0f);
        }
        uint32_t tmask = tri_valid_mask(vmask, K);
        const uint32_t full = (1u << K) - 1u;
        const uint32_t drawn = a.face_mask ? (__ldg(a.face_mask + f0 + tid) & full) : full;
        const unsigned ntri_bad = K - __popc(tmask);   // culled: an invalid vertex
        tmask &= drawn;
        if ((vmask != all || drawn != full) && tmask) {   // bounds over the vertices of drawn triangles only
            mnx = 3.0e38f; mxx = -3.0e38f; mny = 3.0e38f; mxy = -3.0e38f;
            for (int k = 0; k < KV; ++k) {
                if (!vertex_used(tmask, k, K)) continue;
                const DVert d = decide_vertex(cam, df_project(cam, p[3 * k], p[3 * k + 1], p[3 * k + 2]), ox, oy);
                mnx = fminf(mnx, d.xs); mxx = fmaxf(mxx, d.xs);
                mny = fminf(mny, d.ys); mxy = fmaxf(mxy, d.ys);
            }
        }
        if (ntri_bad) atomicAdd(&s_culled, ntri_bad);
        if (a.splat && tmask) {   // (kept for the count pass in the third vertex)
            const float reach = fmaxf(fmaxf(cam.cx - mnx, mxx - cam.cx), fmaxf(cam.cy - mny, mxy - cam.cy));
            const float e = polygon_pad(p, cam, c0.Z.h, fmaxf(reach, 0.0f));
            dec[2].w = e;
            mnx -= e; mxx += e; mny -= e; mxy += e;
        }
        if (tmask) {
            const FanRect r = rect_from_bounds(mnx, mxx, mny, mxy, cam.width, cam.height);
            if (!r.empty) {
                const int tx0 = r.i0 >> tile_shift, tx1 = r.i1 >> tile_shift;
                const int ty0 = r.j0 >> tile_shift, ty1 = r.j1 >> tile_shift;
                const int w = tx1 - tx0 + 1, h = ty1 - ty0 + 1;
                count = (uint32_t)(w * h);
                s_rect[tid][0] = (uint32_t)tx0 | ((uint32_t)ty0 << 16);
                s_rect[tid][1] = (uint32_t)w | ((uint32_t)h << 16);
            }
        }
    }
    // Block-wide exclusive scan of the counts (fan order).
    uint32_t x = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t t = lane < kBinThreads / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < kBinThreads / 32) s_warp[lane] = t;
    }
    __syncthreads();
    const uint32_t incl = x + (warp > 0 ? s_warp[warp - 1] : 0);
    s_off[tid + 1] = incl;
    if (tid == 0) s_off[0] = 0;
    const uint32_t total = s_warp[kBinThreads / 32 - 1];

    // The block's range of the pair array: one atomic reservation.
    if (tid == 0) {
        s_excl = total ? atomicAdd(&st->pairs, (unsigned long long)total) : 0ull;
        if (vid == 0) {
            st->cap = (unsigned long long)cap;
            st->n_tiles = a.n_tiles;
            st->sort_bits = a.sort_bits;
        }
        if (s_culled) atomicAdd(&st->culled, (unsigned long long)s_culled);
    }
    __syncthreads();

    // Output-major emission: consecutive threads write consecutive pairs.
    const unsigned long long base = s_excl;
    for (uint32_t o0 = warp * 32; o0 < total; o0 += kBinThreads) {   // (whole warps take part)
        const uint32_t o = o0 + lane;
        const unsigned long long idx = base + o;
        const bool in = o < total && idx < (unsigned long long)cap;
        uint32_t tile = ~0u;
        int lo = 0;
        if (in) {
            int hi = nloc;   // largest f with s_off[f] <= o
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (s_off[mid] <= o) lo = mid; else hi = mid;
            }
            const uint32_t k = o - s_off[lo];
            const uint32_t r0 = s_rect[lo][0], r1 = s_rect[lo][1];
            const uint32_t w = r1 & 0xFFFFu;
            const uint32_t tx = (r0 & 0xFFFFu) + k % w, ty = (r0 >> 16) + k / w;
            tile = tile_base + ty * tiles_x + tx;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, tile);
        const int leader = __ffs(peers) - 1;
        uint32_t rank = 0;
        if (in && lane == leader) rank = atomicAdd(a.tile_cnt + tile, (uint32_t)__popc(peers));
        rank = __shfl_sync(0xffffffffu, rank, leader) + __popc(peers & ((1u << lane) - 1u));
        if (in) {
            a.pairs[idx] = make_uint2(tile, (uint32_t)(f0 + lo));
            a.ranks[idx] = rank;
        }
    }
}

}  // namespace

cudaError_t launch_bin(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    if (ra.n_fans == 0) return cudaSuccess;
    const size_t smem = sizeof(float) * kBinThreads * (ra.K + 1) * 3;
    cudaFuncSetAttribute(bin_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    BinArgs a;
    a.xyz = ra.xyz;
    a.n_fans = ra.n_fans;
    a.K = ra.K;
    a.tile_shift = 0;
    while ((1 << a.tile_shift) < L.tile) ++a.tile_shift;
    a.cap = L.cap;
    a.fan_blocks = L.bin_fan_blocks;
    a.n_tiles = (unsigned)L.n_tiles;
    a.sort_bits = (unsigned)L.tile_bits;
    a.st = reinterpret_cast<Status *>(ra.ws + L.off_status);
    a.pairs = reinterpret_cast<uint2 *>(ra.ws + L.off_pairs);
    a.ranks = reinterpret_cast<uint32_t *>(ra.ws + L.off_ranks);
    a.tile_cnt = reinterpret_cast<uint32_t *>(ra.ws + L.off_tile_cnt);
    a.vt = ra.vt;
    a.dec = reinterpret_cast<float4 *>(ra.ws + L.off_dec);
    a.V = L.V;
    a.face_mask = ra.splat ? nullptr : ra.prm.face_mask;
    a.splat = ra.splat;
    bin_kernel<<<(unsigned)L.bin_blocks, kBinThreads, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace ms
