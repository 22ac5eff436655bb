// Per-pixel resolve of the fragment buffer: exact depth order and front-to-back
// compositing (forward), and its adjoint (backward).
//
// A pixel's fragment records sit contiguously.  Order: (depth, triangle id), the depth a
// double-float value (high part in the record's first word, low part in its fourth).
// Compositing stops once the transmittance falls below T_eps.
//
// Pixels are resolved by groups of 8, 16 or 32 lanes, by their fragment count, one record a
// lane: the records are read coalesced, a record's place is the number of records before it,
// counted against the group's keys in shared memory, and the composite's products and sums run
// over the sorted values in front-to-back order, each rounded as a sequential composite rounds
// it.  A warp takes a deeper pixel alone: up to 64 records are placed at once and composited in
// two rounds of 32; beyond that, every pass over the records keeps the 32 nearest beyond the last
// composited one (merging 32 records at a time), so the order is exact for any depth complexity.
// A round after the first counts as an extra pass.
//
// pixel_alloc_kernel (tiles.cu) lists the pixels by class of fragment count, spans of 1024 pixel
// slots in descending count, so a warp's groups run loops of about the same length on
// neighbouring records.  Warps take units of the lists in turn and fetch the next units' entries
// and counts while they work.
//
// The forward also records, per pixel, the record index of each committed fragment in
// commit order (and where they end early).  The backward walks that list (no sorting), and at
// each committed fragment f forms, from the recomputed transmittance T_f,
// dC/dc_f = T_f a_f, dC/da_f = T_f c_f - (C_out - C_{<=f}) / (1 - a_f) and
// dA/da_f = T_out / (1 - a_f).  It writes dL/dc_f and dL/da_f, with the fragment's
// triangle and pixel, as an adjoint record (the pixel's c-th composited fragment in slot
// c of its record range); the chain pass (chain.cu) takes them to the vertices record by
// record, so this pass does no atomics.
//
// What bounds them: the forward issues on two thirds of its cycles and waits on scattered
// record reads otherwise (1M fans at 1080p, 10.4M fragments: 0.26 ms; one thread a pixel with a
// sorted register buffer, 114 registers and 11 of 32 lanes active: 0.54 ms).  The backward
// waits on its record reads (0.19 ms there, 72 long-scoreboard cycles an instruction).
#include "raster_common.cuh"

namespace ms {

namespace {

constexpr uint32_t kEnd = 0xffffffffu;

struct ResolveArgs {
    int64_t npx;
    const float4 *frags;
    float T_eps, bg0, bg1, bg2;
    Status *st;
    float *tfinal;
    float4 *adj;               // backward: per composited fragment, in commit order within the
                               // pixel's record range: (dL/dc * T a, dL/da), (triangle, pixel, 0, 0)
                               // (32 bytes, whole sectors: 16 + 8 bytes in two arrays took twice as long)
    uint32_t *corder;          // per pixel: record indices in commit order (same offsets as records), then
                               // kEnd if fewer were composited than there are records
    // pixels whose fragments have records: list_b holds those of more than 16 (more than 32 from its
    // end, the others from its start), list_a the others with their record offsets (9 to 16 from
    // its end, 1 to 8 from its start); st->classes counts the four
    const uint2 *list_a;
    const uint32_t *list_b, *offsets;
    int64_t order_b;           // entries of list_b (list_a: npx)
    const uint32_t *counts;
    ViewTable vt;
};

// The work of the resolve kernel: warps take units of the pixel lists in turn, a unit being
// one pixel of more than 16 records, two of 9 to 16 or four of 1 to 8.
constexpr int kGroupThreads = 256, kResident = 4;   // threads a block, blocks a multiprocessor
struct Units {
    uint32_t c16, c8;             // pixels of 9 to 16 and of 1 to 8 records
    uint32_t deep, n32, n16, n8;  // unit bounds of the classes
    __device__ __forceinline__ Units(const ResolveArgs &a) {
        const uint4 c = *reinterpret_cast<const uint4 *>(a.st->classes);
        deep = c.x;
        n32 = deep + c.y;
        c16 = c.z;
        c8 = c.w;
        n16 = n32 + (c16 + 1) / 2;
        n8 = n16 + (c8 + 3) / 4;
    }
    // This lane's entry of unit u (pixel and, from list_a, its record offset; no pixel: ~0).
    __device__ __forceinline__ uint2 entry(const ResolveArgs &a, int64_t u, int lane) const {
        uint2 e = make_uint2(~0u, 0u);
        if (u < deep) {
            e.x = __ldg(a.list_b + (a.order_b - 1 - u));
        } else if (u < n32) {
            e.x = __ldg(a.list_b + (u - deep));
        } else if (u < n16) {
            const int64_t q = 2 * (u - n32) + (lane >> 4);
            if (q < c16) e = __ldg(a.list_a + (a.npx - 1 - q));
        } else if (u < n8) {
            const int64_t q = 4 * (u - n16) + (lane >> 3);
            if (q < c8) e = __ldg(a.list_a + q);
        }
        return e;
    }
};

// A pixel with its records (all of which the buffer holds); count 0 where there is none.
struct Pixel {
    uint32_t pix, off, n;
};
__device__ __forceinline__ Pixel pixel_of(const ResolveArgs &a, const uint2 e, bool from_b) {
    Pixel p = {e.x, e.y, 0u};
    if (e.x < (uint64_t)a.npx) {
        p.n = __ldg(a.counts + e.x);
        if (from_b) p.off = __ldg(a.offsets + e.x);
    }
    return p;
}
__device__ __forceinline__ bool is_pixel(const ResolveArgs &a, const Pixel &p) { return p.pix < (uint64_t)a.npx; }

// Shared words of one warp: sort keys and ids by record, then the values in sorted places.
struct GroupMem {
    unsigned long long key[64];
    float oma[64], w[64], c[3][64];   // 1 - opacity, T a, colour
    uint32_t tri[64], src[64];        // tie-break id, record of each place
};

// Depths are positive: their bits order like their values; the low part (either sign, zeros
// alike) maps to an unsigned order.
__device__ __forceinline__ unsigned long long sort_key(const float4 &r0) {
    const uint32_t lb = __float_as_uint(r0.w + 0.0f);
    return (unsigned long long)__float_as_uint(r0.x) << 32 | ((lb & 0x80000000u) ? ~lb : (lb | 0x80000000u));
}

__device__ __forceinline__ void put(GroupMem &m, int at, bool has, const float4 &r1, uint32_t src) {
    m.oma[at] = has ? 1.0f - r1.w : 1.0f;
    m.w[at] = has ? r1.w : 0.0f;
    m.c[0][at] = r1.x;
    m.c[1][at] = r1.y;
    m.c[2][at] = r1.z;
    m.src[at] = src;
}

// Transmittance in front of place `sub` (T0 in front of place 0), multiplied front to back.
__device__ __forceinline__ float front_product(const float *oma, int sub, int nmax, float T0) {
    float T = T0;
    const float4 *op = reinterpret_cast<const float4 *>(oma);
    for (int i = 0; i < nmax; i += 4) {
        const float4 o = op[i >> 2];
        if (i < sub) T *= o.x;
        if (i + 1 < sub) T *= o.y;
        if (i + 2 < sub) T *= o.z;
        if (i + 3 < sub) T *= o.w;
    }
    return T;
}

// Composites the n <= G sorted places from g0 on (n <= nmax for every group of the warp) behind
// transmittance T and the sums C (this lane's channel: sub % 4, the fourth idle); sets T to the
// transmittance behind them and returns the number composited before T < T_eps (ended then set).
template <int G>
__device__ __forceinline__ int composite(GroupMem &m, int g0, int at0, int n, int nmax, float T_eps, float &T, float &C,
                                         bool &ended) {
    const int sub = (threadIdx.x & 31) - g0;
    const int at = at0 + sub;
    const float Tl = front_product(m.oma + at0, sub, nmax, T);
    const float Tn = Tl * m.oma[at];
    const uint32_t low = (__ballot_sync(0xffffffffu, sub < n && Tn < T_eps) >> g0) &
                         (G == 32 ? 0xffffffffu : (1u << (G & 31)) - 1u);
    ended = low != 0u;
    const int ncom = ended ? __ffs(low) : n;
    m.w[at] = sub < ncom ? Tl * m.w[at] : 0.0f;
    if (sub >= ncom) m.c[0][at] = m.c[1][at] = m.c[2][at] = 0.0f;
    __syncwarp();
    const int ch = min(sub & 3, 2);
    const float4 *wp = reinterpret_cast<const float4 *>(m.w + at0);
    const float4 *cp = reinterpret_cast<const float4 *>(m.c[ch] + at0);
    for (int i = 0; i < nmax; i += 4) {
        const float4 x = wp[i >> 2], y = cp[i >> 2];
        C += x.x * y.x;
        C += x.y * y.y;
        C += x.z * y.z;
        C += x.w * y.w;
    }
    const float Tf = __shfl_sync(0xffffffffu, Tn, g0 + max(ncom - 1, 0));
    if (n > 0) T = Tf;
    return ncom;
}

__device__ __forceinline__ void write_pixel(const ResolveArgs &a, const Pixel &e, float T, float C0, float C1, float C2,
                                            uint32_t ncom) {
    const ViewDev &vw = a.vt.v[view_of_pixel(a.vt, (unsigned long long)e.pix)];
    reinterpret_cast<float4 *>(vw.out)[(int64_t)e.pix - (int64_t)vw.pix_base] =
        make_float4(C0 + T * a.bg0, C1 + T * a.bg1, C2 + T * a.bg2, 1.0f - T);
    a.tfinal[e.pix] = T;
    if (ncom < e.n) a.corder[(size_t)e.off + ncom] = kEnd;
}

// One warp's 32 / G pixels (e per group); returns the fragments composited (first lanes).
template <int G>
__device__ __forceinline__ uint32_t resolve_group(const ResolveArgs &a, GroupMem &m, const Pixel e) {
    const int lane = threadIdx.x & 31, sub = lane & (G - 1), g0 = lane & ~(G - 1);
    const bool valid = is_pixel(a, e);
    const int64_t off = e.off;
    const int n = e.n <= (uint32_t)G ? (int)e.n : 0;   // (it is: a bound the loops below are unrolled by)
    const int nmax = __reduce_max_sync(0xffffffffu, n);
    const bool has = sub < n;
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
    if (has) ld_rec(a.frags + (size_t)kRecFwd * (size_t)(off + sub), r0, r1);
    const unsigned long long key = has ? sort_key(r0) : ~0ull;
    __syncwarp();   // the words are still read for the previous unit
    m.key[lane] = key;
    __syncwarp();
    int rank = 0;
    const ulonglong2 *kp = reinterpret_cast<const ulonglong2 *>(m.key + g0);
    for (int i = 0; i < nmax; i += 2) {
        const ulonglong2 k = kp[i >> 1];
        rank += (int)(k.x < key) + (int)(k.y < key);
    }
    // equal depths leave two records on one place: then the triangle id decides
    const uint32_t placed = __reduce_or_sync(0xffffffffu, has ? 1u << (g0 + rank) : 0u);
    if (placed != __ballot_sync(0xffffffffu, has)) {
        const uint32_t tri = __float_as_uint(r0.y);
        m.tri[lane] = tri;
        __syncwarp();
        rank = 0;
        for (int i = 0; i < nmax; ++i) {
            const unsigned long long k = m.key[g0 + i];
            rank += (int)(k < key || (k == key && i < n && m.tri[g0 + i] < tri));
        }
    }
    put(m, g0 + (has ? rank : sub), has, r1, (uint32_t)sub);   // (the other lanes fill the places past n)
    __syncwarp();
    float T = 1.0f, C = 0.0f;
    bool ended;
    const int ncom = composite<G>(m, g0, g0, n, nmax, a.T_eps, T, C, ended);
    const float C1 = __shfl_sync(0xffffffffu, C, g0 + 1), C2 = __shfl_sync(0xffffffffu, C, g0 + 2);
    if (valid && sub < ncom) a.corder[off + sub] = m.src[lane];
    if (valid && sub == 0) write_pixel(a, e, T, C, C1, C2, (uint32_t)ncom);
    return valid && sub == 0 ? (uint32_t)ncom : 0u;
}

// Places two records a lane (keys ka, kb; ~0: none) among the warp's 64 by (key, id).
__device__ __forceinline__ void place64(GroupMem &m, unsigned long long ka, uint32_t ta, unsigned long long kb,
                                        uint32_t tb, int &ra, int &rb) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    m.key[lane] = ka;
    m.key[lane + 32] = kb;
    m.tri[lane] = ta;
    m.tri[lane + 32] = tb;
    __syncwarp();
    ra = rb = 0;
    const ulonglong2 *kp = reinterpret_cast<const ulonglong2 *>(m.key);
    for (int i = 0; i < 32; ++i) {
        const ulonglong2 k = kp[i];
        ra += (int)(k.x < ka) + (int)(k.y < ka);
        rb += (int)(k.x < kb) + (int)(k.y < kb);
    }
    const bool ha = ka != ~0ull, hb = kb != ~0ull;
    const int n = __popc(__ballot_sync(0xffffffffu, ha)) + __popc(__ballot_sync(0xffffffffu, hb));
    const uint32_t p0 = __reduce_or_sync(0xffffffffu, (ha && ra < 32 ? 1u << ra : 0u) | (hb && rb < 32 ? 1u << rb : 0u));
    const uint32_t p1 = __reduce_or_sync(0xffffffffu, (ha && ra >= 32 ? 1u << (ra - 32) : 0u) |
                                                          (hb && rb >= 32 ? 1u << (rb - 32) : 0u));
    if (__popc(p0) + __popc(p1) != n) {   // equal depths: the id decides
        ra = rb = 0;
        for (int i = 0; i < 64; ++i) {
            const unsigned long long k = m.key[i];
            const uint32_t t = m.tri[i];
            ra += (int)(k < ka || (k == ka && t < ta));
            rb += (int)(k < kb || (k == kb && t < tb));
        }
    }
    __syncwarp();
}

// One warp's pixel of any number of records.
__device__ uint32_t resolve_deep(const ResolveArgs &a, GroupMem &m, const Pixel e) {
    const int lane = threadIdx.x & 31;
    if (!is_pixel(a, e)) return 0;
    const int64_t off = e.off;
    const int n = (int)e.n;
    const float4 *rec = a.frags + (size_t)kRecFwd * (size_t)off;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float T = 1.0f, C = 0.0f;
    uint32_t ncom = 0, extra = 0;
    bool ended = false;
    if (n <= 64) {
        const bool ha = lane < n, hb = lane + 32 < n;
        float4 a0 = zero, a1 = zero, b0 = zero, b1 = zero;
        if (ha) ld_rec(rec + kRecFwd * lane, a0, a1);
        if (hb) ld_rec(rec + kRecFwd * (lane + 32), b0, b1);
        int ra, rb;
        place64(m, ha ? sort_key(a0) : ~0ull, __float_as_uint(a0.y), hb ? sort_key(b0) : ~0ull, __float_as_uint(b0.y),
                ra, rb);
        put(m, ha ? ra : lane, ha, a1, (uint32_t)lane);
        put(m, hb ? rb : lane + 32, hb, b1, (uint32_t)lane + 32u);   // (places past n lie in the upper half)
        __syncwarp();
        for (int at = 0; at < n && !ended; at += 32) {
            const int k = min(n - at, 32);
            const int c = composite<32>(m, 0, at, k, k, a.T_eps, T, C, ended);
            if (lane < c) a.corder[off + ncom + lane] = m.src[at + lane];
            ncom += c;
            extra += at ? 1u : 0u;
        }
    } else {
        unsigned long long last_k = 0;   // the last composited record; depths are > 0
        uint32_t last_t = 0;
        for (bool more = true; more && !ended; extra += more && !ended) {
            // the 32 nearest records beyond the last composited one
            unsigned long long bk = ~0ull;
            uint32_t bt = 0xffffffffu, bs = 0;
            more = false;
            for (int i0 = 0; i0 < n; i0 += 32) {
                const int i = i0 + lane;
                unsigned long long k = ~0ull;
                uint32_t t = 0xffffffffu;
                if (i < n) {
                    const float4 r0 = rec[kRecFwd * i];
                    const unsigned long long kk = sort_key(r0);
                    const uint32_t tt = __float_as_uint(r0.y);
                    if (kk > last_k || (kk == last_k && tt > last_t)) {
                        k = kk;
                        t = tt;
                    }
                }
                int ra, rb;
                place64(m, bk, bt, k, t, ra, rb);
                // (records that are not there tie behind all others: they go past them in any order)
                if (bk != ~0ull) { m.key[ra] = bk; m.tri[ra] = bt; m.src[ra] = bs; }
                if (k != ~0ull) { m.key[rb] = k; m.tri[rb] = t; m.src[rb] = (uint32_t)i; }
                const int live = __popc(__ballot_sync(0xffffffffu, bk != ~0ull)) + __popc(__ballot_sync(0xffffffffu, k != ~0ull));
                more |= live > 32;
                __syncwarp();
                bk = lane < live ? m.key[lane] : ~0ull;
                bt = lane < live ? m.tri[lane] : 0xffffffffu;
                bs = lane < live ? m.src[lane] : 0u;
            }
            const bool has = bk != ~0ull;
            const int k = __popc(__ballot_sync(0xffffffffu, has));
            if (k == 0) break;
            __syncwarp();
            put(m, lane, has, has ? rec[kRecFwd * bs + 1] : zero, bs);
            __syncwarp();
            const int c = composite<32>(m, 0, 0, k, k, a.T_eps, T, C, ended);
            if (lane < c) a.corder[off + ncom + lane] = bs;
            ncom += c;
            last_k = __shfl_sync(0xffffffffu, bk, k - 1);
            last_t = __shfl_sync(0xffffffffu, bt, k - 1);
        }
    }
    const float C1 = __shfl_sync(0xffffffffu, C, 1), C2 = __shfl_sync(0xffffffffu, C, 2);
    if (lane == 0) {
        write_pixel(a, e, T, C, C1, C2, ncom);
        if (extra) atomicAdd(&a.st->extra_passes, (unsigned long long)extra);
    }
    return lane == 0 ? ncom : 0u;
}

__global__ void __launch_bounds__(kGroupThreads, kResident) resolve_kernel(const __grid_constant__ ResolveArgs a) {
    __shared__ __align__(16) GroupMem s_mem[kGroupThreads / 32];
    const Units U(a);
    GroupMem &m = s_mem[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (kGroupThreads / 32);
    uint32_t ncom = 0;
    int64_t u = (int64_t)blockIdx.x * (kGroupThreads / 32) + (threadIdx.x >> 5);
    // entries are fetched two units ahead, counts one unit ahead
    Pixel e1 = pixel_of(a, U.entry(a, u, lane), u < U.n32);
    uint2 e2 = U.entry(a, u + warps, lane);
    for (; u < U.n8; u += warps) {
        const Pixel e = e1;
        e1 = pixel_of(a, e2, u + warps < U.n32);
        e2 = U.entry(a, u + 2 * warps, lane);
        if (u < U.deep)
            ncom += resolve_deep(a, m, e);
        else if (u < U.n32)
            ncom += resolve_group<32>(a, m, e);
        else if (u < U.n16)
            ncom += resolve_group<16>(a, m, e);
        else
            ncom += resolve_group<8>(a, m, e);
    }
    ncom = __reduce_add_sync(0xffffffffu, ncom);
    if (lane == 0 && ncom) atomicAdd(&a.st->commits, (unsigned long long)ncom);
}

// Backward, one thread a pixel of the lists (a warp's lanes run loops of about the same
// length): no sorting is left, so a lane's sequential walk takes far fewer instructions than the
// groups' prefix sums (measured: 0.26 against 0.34 ms on 10.4M fragments).  The walk waits on
// its records, so the record after the next one's index and the next record load while the
// current one is worked on.
constexpr int kBwdThreads = 64;
__global__ void __launch_bounds__(kBwdThreads) resolve_bwd_kernel(const __grid_constant__ ResolveArgs a) {
    const int64_t q = (int64_t)blockIdx.x * kBwdThreads + threadIdx.x;
    const uint4 cl = *reinterpret_cast<const uint4 *>(a.st->classes);
    const int64_t n0 = cl.x, n1 = n0 + cl.y, n2 = n1 + cl.z;
    if (q >= n2 + cl.w) return;
    uint2 entry = make_uint2(0u, 0u);
    if (q < n0)
        entry.x = __ldg(a.list_b + (a.order_b - 1 - q));
    else if (q < n1)
        entry.x = __ldg(a.list_b + (q - n0));
    else
        entry = __ldg(q < n2 ? a.list_a + (a.npx - 1 - (q - n1)) : a.list_a + (q - n2));
    const Pixel e = pixel_of(a, entry, q < n1);
    if (!is_pixel(a, e)) return;
    const int64_t off = e.off;
    const uint32_t n = e.n;
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float4 *adj = a.adj + 2 * off;
    const ViewDev &vw = a.vt.v[view_of_pixel(a.vt, (unsigned long long)e.pix)];
    const int64_t lpix = (int64_t)e.pix - (int64_t)vw.pix_base;
    const float4 *rec = a.frags + (size_t)kRecFwd * off;
    const uint32_t *ord = a.corder + off;
    const float4 g = reinterpret_cast<const float4 *>(vw.dL)[lpix];
    const float4 ov = reinterpret_cast<const float4 *>(vw.out_fwd)[lpix];
    const float Tout = a.tfinal[e.pix];
    float T = 1.0f, C0 = 0.0f, C1 = 0.0f, C2 = 0.0f;
    // (indices past the last composited fragment are not read as records)
    uint32_t i1 = ord[0], i2 = n > 1 ? ord[1] : kEnd;
    float4 id1 = zero, col1 = zero;
    if (i1 < n) ld_rec(rec + (size_t)kRecFwd * i1, id1, col1);
    uint32_t c = 0;
    for (; c < n && i1 < n; ++c) {
        const float tri = id1.y;
        const float4 col = col1;
        if (i2 < n) ld_rec(rec + (size_t)kRecFwd * i2, id1, col1);
        i1 = i2;
        i2 = c + 2 < n && i2 < n ? ord[c + 2] : kEnd;
        const float al = col.w;
        const float w = T * al;
        const float nC0 = C0 + w * col.x, nC1 = C1 + w * col.y, nC2 = C2 + w * col.z;
        const float inv = 1.0f / fmaxf(1.0f - al, 1e-6f);
        const float ga = g.x * (T * col.x - (ov.x - nC0) * inv) + g.y * (T * col.y - (ov.y - nC1) * inv) +
                         g.z * (T * col.z - (ov.z - nC2) * inv) + g.w * Tout * inv;
        st_rec(adj + 2 * c, make_float4(g.x * w, g.y * w, g.z * w, ga), make_float4(tri, __uint_as_float(e.pix), 0.0f, 0.0f));
        C0 = nC0; C1 = nC1; C2 = nC2;
        T *= (1.0f - al);
    }
    // slots past the composited fragments carry a zero gradient (the chain pass reads
    // every slot of the pixel's range)
    for (; c < n; ++c) st_rec(adj + 2 * c, zero, zero);
}

__global__ void grad_scatter_kernel(const float4 *__restrict__ g, int64_t V, float *__restrict__ dx,
                                    float *__restrict__ dc, float *__restrict__ da) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
        float4 a, b;
        ld_rec(g + 2 * v, a, b);
        dx[3 * v] += a.x;
        dx[3 * v + 1] += a.y;
        dx[3 * v + 2] += a.z;
        da[v] += a.w;
        dc[3 * v] += b.x;
        dc[3 * v + 1] += b.y;
        dc[3 * v + 2] += b.z;
    }
}

}  // namespace

namespace {

ResolveArgs make_args(const RenderArgs &ra) {
    const RenderLayout &L = ra.L;
    ResolveArgs a;
    a.npx = L.npx;
    a.frags = reinterpret_cast<const float4 *>(ra.ws + L.off_frags);
    a.T_eps = ra.prm.T_eps;
    a.bg0 = ra.prm.bg[0];
    a.bg1 = ra.prm.bg[1];
    a.bg2 = ra.prm.bg[2];
    a.st = reinterpret_cast<Status *>(ra.ws + L.off_status);
    a.tfinal = reinterpret_cast<float *>(ra.ws + L.off_tfinal);
    a.adj = reinterpret_cast<float4 *>(ra.ws + L.off_adj);
    a.corder = reinterpret_cast<uint32_t *>(ra.ws + L.off_corder);
    a.list_a = reinterpret_cast<const uint2 *>(ra.ws + L.off_order_a);
    a.list_b = reinterpret_cast<const uint32_t *>(ra.ws + L.off_order_b);
    a.offsets = reinterpret_cast<const uint32_t *>(ra.ws + L.off_offsets);
    a.order_b = L.order_b;
    a.counts = reinterpret_cast<const uint32_t *>(ra.ws + L.off_counts);
    a.vt = ra.vt;
    return a;
}

}  // namespace

cudaError_t launch_resolve(const RenderArgs &ra, bool backward, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    if (L.npx == 0) return cudaSuccess;
    // the classes' sizes are known on the device only: a persistent grid of the resident blocks,
    // at most one warp a pixel
    const unsigned grid = (unsigned)min64((L.npx + kGroupThreads / 32 - 1) / (kGroupThreads / 32), 152 * kResident);
    if (backward)
        resolve_bwd_kernel<<<(unsigned)((L.npx + kBwdThreads - 1) / kBwdThreads), kBwdThreads, 0, st>>>(
            make_args(ra));
    else
        resolve_kernel<<<grid, kGroupThreads, 0, st>>>(make_args(ra));
    return cudaGetLastError();
}

cudaError_t launch_grad_scatter(const RenderArgs &ra, cudaStream_t st) {
    const RenderLayout &L = ra.L;
    if (L.V == 0) return cudaSuccess;
    const int grid = (int)min64((L.V + 255) / 256, 16 * 152);
    grad_scatter_kernel<<<grid, 256, 0, st>>>(reinterpret_cast<const float4 *>(ra.ws + L.off_grad), L.V, ra.d_xyz,
                                              ra.d_rgb, ra.d_alpha);
    return cudaGetLastError();
}

}  // namespace ms
