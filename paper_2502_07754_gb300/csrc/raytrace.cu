// Ray tracing of the triangle soup with shadows (the paper's motivation for the mesh form,
// Sec. 1 and its discussion of ray-traced Gaussian renderers: a triangle soup is what ray
// tracers take, with secondary effects such as shadows).  The paper gives no shading
// model; the one implemented (also the oracle's):
//   * primary rays: the pixel-centre ray of the pinhole camera, x = C + t d with d of unit
//     view depth (so t is the view depth); every triangle it crosses at t > znear is a
//     fragment with the ray's barycentrics (equal to the rasteriser's perspective-correct
//     ones), ordered by t, ties by triangle index, composited front to back as the raster
//     does (C += T a c, T *= 1 - a; out = (C + T bg, 1 - T));
//   * shadows: a point light L; a fragment at p gets the transmittance S, the product of
//     (1 - a_g) over every other triangle g the segment p -> L crosses (parameter strictly
//     inside (1e-9, 1 - 1e-9)), and its colour becomes c (k + (1 - k) S), k the ambient
//     share; a shadow ray stops once S < T_eps, the primary composite's own bound.
// Intersections are decided as in FP64 (Moller-Trumbore, edges closed).
//
// Acceleration: a linear BVH (Karras 2012, "Maximizing parallelism in the construction of
// BVHs, octrees, and k-d trees"): 30-bit Morton codes of the triangle centroids in the
// scene box, sorted (with the triangle index as the low 32 bits, so every key is unique)
// by the library's radix sort; every internal node finds its key range and split from the
// longest common prefixes of its neighbours; boxes are merged bottom-up, the second of a
// node's two children to arrive computing the node (an atomic counter per node, no waits).
// Boxes are the binary32 vertex bounds widened by a small margin so that the binary32
// slab test never rejects a box the FP64 ray meets.
//
// Tracing gathers a ray's crossings in passes: each pass walks the BVH keeping the KB
// nearest crossings beyond the last composited one (by (t, triangle)), composites them in
// order, and repeats while some crossing was left out and the transmittance is above
// T_eps.  A pass skips boxes that end before the last composited crossing and, once its
// buffer is full, boxes that start beyond the farthest kept one.  FP64 runs at a small fraction
// of the binary32 rate here, so a triangle meets a binary32 filter (mt_may_hit) before the exact
// test. A ray takes that in FP64, which also orders and weighs its crossings. A segment to the light
// takes it in double-float (mt_df), and in FP64 only where that is not certain (the segment within
// 2^-40 of an edge): its crossings are FP64's, its factors within 2^-42 of them.
#include "ms_common.cuh"
#include "ms_internal.h"

namespace ms {

namespace {

constexpr int kBvhThreads = 256;
constexpr int kTracePix = 32;      // pixels a block (8 x 4, one warp)
constexpr int kTraceWarps = 4;     // and the warps that trace their segments to the light
constexpr int kPlainWarps = 2;     // without shadows: warps of 8 x 4 pixels a block
// Crossings that a pass keeps (1.6M triangles at 800x800: 8, 16, 24, 32 take 45, 39, 42, 43 ms with
// shadows and 8.7, 6.9, 5.9, 6.1 ms without).
template <bool SHADOWS>
constexpr int kTraceKB = SHADOWS ? 16 : 24;
constexpr int kStack = 64;
constexpr int kWalkShare = 1;   // a warp leaves the tree when at most this many of its lanes walk for each that waits
constexpr int kTraceBlocks = 5;    // blocks an SM with shadows

constexpr double kSegEps = 1e-9;

// An internal node holds its children's boxes (low corner, high corner), so a traversal step waits
// for one 64-byte read.
struct alignas(16) BvhNode {
    float box[2][6];
    int child[2];      // < n - 1 internal, >= n - 1 leaf (n - 1 + sorted position)
    int pad[2];
};

struct BvhLayout {
    size_t nodes, parent, flags, leaf_tri, keys0, keys1, bounds, status, scratch, total;
};

size_t al256(size_t x) { return (x + 255) / 256 * 256; }

BvhLayout bvh_layout(int64_t T) {
    BvhLayout L;
    const int64_t n = T > 0 ? T : 1;
    size_t o = 0;
    L.status = o;   o = al256(o + 256);
    L.bounds = o;   o = al256(o + 8 * sizeof(unsigned));
    L.nodes = o;    o = al256(o + (size_t)n * sizeof(BvhNode));   // (n - 1 internal nodes)
    L.parent = o;   o = al256(o + (size_t)(2 * n - 1) * 4);
    L.flags = o;    o = al256(o + (size_t)n * 4);
    L.leaf_tri = o; o = al256(o + (size_t)n * 4);
    L.keys0 = o;    o = al256(o + (size_t)n * 8);
    L.keys1 = o;    o = al256(o + (size_t)n * 8);
    L.scratch = o;  o = al256(o + sort_scratch_bytes(n, 4));
    L.total = o;
    return L;
}

// Vertex indices of triangle t: explicit, or the implicit fan topology of K triangles a fan.
__device__ __forceinline__ void tri_verts(const int32_t *tris, int K, int64_t t, int64_t v[3]) {
    if (tris) {
        v[0] = __ldg(tris + 3 * t);
        v[1] = __ldg(tris + 3 * t + 1);
        v[2] = __ldg(tris + 3 * t + 2);
    } else {
        const int64_t g = t / K;
        const int j = (int)(t - g * K);
        const int64_t c = g * (K + 1);
        v[0] = c;
        v[1] = c + 1 + j;
        v[2] = c + 1 + (j + 1 == K ? 0 : j + 1);
    }
}

// Floats ordered as unsigned integers (for atomic min / max of the scene box).
__device__ __forceinline__ unsigned f2o(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float o2f(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

__global__ void bounds_init_kernel(unsigned *b) {
    if (threadIdx.x < 3) b[threadIdx.x] = 0xffffffffu;   // min
    else if (threadIdx.x < 6) b[threadIdx.x] = 0u;        // max
}

__global__ void __launch_bounds__(kBvhThreads) centroid_bounds_kernel(const float *__restrict__ xyz,
                                                                      const int32_t *__restrict__ tris, int K,
                                                                      int64_t T, unsigned *b) {
    float lo[3] = {3.0e38f, 3.0e38f, 3.0e38f}, hi[3] = {-3.0e38f, -3.0e38f, -3.0e38f};
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += (int64_t)gridDim.x * blockDim.x) {
        int64_t v[3];
        tri_verts(tris, K, t, v);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float c = (__ldg(xyz + 3 * v[0] + r) + __ldg(xyz + 3 * v[1] + r) + __ldg(xyz + 3 * v[2] + r)) *
                             (1.0f / 3.0f);
            lo[r] = fminf(lo[r], c);
            hi[r] = fmaxf(hi[r], c);
        }
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[r] = fminf(lo[r], __shfl_xor_sync(0xffffffffu, lo[r], o));
            hi[r] = fmaxf(hi[r], __shfl_xor_sync(0xffffffffu, hi[r], o));
        }
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            atomicMin(&b[r], f2o(lo[r]));
            atomicMax(&b[3 + r], f2o(hi[r]));
        }
    }
}

// 10 bits of x spread to every third bit.
__device__ __forceinline__ unsigned long long spread3(unsigned x) {
    unsigned long long v = x & 0x3ffu;
    v = (v | (v << 16)) & 0x030000FFull;
    v = (v | (v << 8)) & 0x0300F00Full;
    v = (v | (v << 4)) & 0x030C30C3ull;
    v = (v | (v << 2)) & 0x09249249ull;
    return v;
}

__global__ void __launch_bounds__(kBvhThreads) morton_kernel(const float *__restrict__ xyz,
                                                             const int32_t *__restrict__ tris, int K, int64_t T,
                                                             const unsigned *__restrict__ b,
                                                             unsigned long long *__restrict__ keys) {
    float lo[3], ext[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        lo[r] = o2f(b[r]);
        const float e = o2f(b[3 + r]) - lo[r];
        ext[r] = e > 0.0f ? e : 1.0f;
    }
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += (int64_t)gridDim.x * blockDim.x) {
        int64_t v[3];
        tri_verts(tris, K, t, v);
        unsigned long long code = 0;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float c = (__ldg(xyz + 3 * v[0] + r) + __ldg(xyz + 3 * v[1] + r) + __ldg(xyz + 3 * v[2] + r)) *
                            (1.0f / 3.0f);
            const float q = fminf(fmaxf((c - lo[r]) / ext[r] * 1024.0f, 0.0f), 1023.0f);
            code |= spread3((unsigned)q) << (2 - r);
        }
        keys[t] = (code << 32) | (unsigned long long)(uint32_t)t;
    }
}

// Common prefix length of sorted keys i and j (-1 outside [0, n)).
__device__ __forceinline__ int delta(const unsigned long long *k, int64_t n, int64_t i, int64_t j) {
    if (j < 0 || j >= n) return -1;
    return __clzll(k[i] ^ k[j]);
}

__global__ void __launch_bounds__(kBvhThreads) radix_tree_kernel(const unsigned long long *__restrict__ keys,
                                                                 int64_t n, BvhNode *__restrict__ nodes,
                                                                 uint32_t *__restrict__ parent,
                                                                 int *__restrict__ leaf_tri) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        leaf_tri[i] = (int)(uint32_t)keys[i];
        if (i >= n - 1) continue;
        const int d = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
        const int dmin = delta(keys, n, i, i - d);
        int64_t lmax = 2;
        while (delta(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;   // at most log2(n) + 1 doublings
        int64_t l = 0;
        for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
            if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
        const int64_t j = i + l * d;
        const int dnode = delta(keys, n, i, j);
        int64_t s = 0;
        for (int64_t t = (l + 1) >> 1;; t = (t + 1) >> 1) {
            if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
            if (t == 1) break;
        }
        const int64_t split = i + s * d + (d < 0 ? -1 : 0);
        const int64_t lo = i < j ? i : j, hi = i < j ? j : i;
        const int left = lo == split ? (int)(n - 1 + split) : (int)split;
        const int right = hi == split + 1 ? (int)(n - 1 + split + 1) : (int)(split + 1);
        nodes[i].child[0] = left;
        nodes[i].child[1] = right;
        parent[left] = 2u * (uint32_t)i;        // and which child of it
        parent[right] = 2u * (uint32_t)i + 1u;
    }
}

__global__ void __launch_bounds__(kBvhThreads) bounds_up_kernel(const float *__restrict__ xyz,
                                                                const int32_t *__restrict__ tris, int K, int64_t n,
                                                                BvhNode *nodes, const uint32_t *__restrict__ parent,
                                                                const int *__restrict__ leaf_tri, int *flags) {
    if (n < 2) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t v[3];
        tri_verts(tris, K, leaf_tri[i], v);
        float box[6];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float a = __ldg(xyz + 3 * v[0] + r), b = __ldg(xyz + 3 * v[1] + r), c = __ldg(xyz + 3 * v[2] + r);
            const float lo = fminf(fminf(a, b), c), hi = fmaxf(fmaxf(a, b), c);
            const float m = 1e-5f * (hi - lo) + 1e-6f * fmaxf(fabsf(lo), fabsf(hi)) + 1e-30f;
            box[r] = lo - m;
            box[3 + r] = hi + m;
        }
        int64_t node = n - 1 + i;
        // every child writes its box into its parent; the second to arrive takes both on
        for (int steps = 0; node != 0 && steps < 64 + 64; ++steps) {
            const uint32_t ps = parent[node], p = ps >> 1, side = ps & 1u;
            volatile float *mine = nodes[p].box[side];
#pragma unroll
            for (int r = 0; r < 6; ++r) mine[r] = box[r];
            __threadfence();
            if (atomicAdd(&flags[p], 1) == 0) break;
            __threadfence();
            const volatile float *other = nodes[p].box[side ^ 1u];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                box[r] = fminf(box[r], other[r]);
                box[3 + r] = fmaxf(box[3 + r], other[3 + r]);
            }
            node = p;
        }
    }
}

// ------------------------------------------------------------------------------ tracing

struct TraceArgs {
    const float *xyz, *rgb, *alpha;
    const int32_t *tris;
    int K;
    int64_t T;
    const BvhNode *nodes;
    const int *leaf_tri;
    CamDev cam;
    float Lf[3];       // the light
    int shadows;
    double ambient;
    double T_eps;
    float T_epsf;      // the same
    float bg[3];
    float *out;
    unsigned *overflow;   // traversal stack overflows (status)
};

// A ray's crossing: `at` is the place of its barycentrics, which stay where they are while a pass sorts the
// crossings (moving all of it took 4% longer without a light).
struct alignas(16) Hit {
    double t;
    int tri, at;
};
// A segment's (whose order does not matter).
struct SegHit {
    dfl t, u, v;
};

// Moller-Trumbore in FP64, edges closed: the crossing of o + t d with triangle (P0, P1, P2).
__device__ __noinline__ bool mt(const double o[3], const double d[3], const double P0[3], const double P1[3],
                                const double P2[3], double &t, double &u, double &v) {
    const double e1[3] = {P1[0] - P0[0], P1[1] - P0[1], P1[2] - P0[2]};
    const double e2[3] = {P2[0] - P0[0], P2[1] - P0[1], P2[2] - P0[2]};
    const double pv[3] = {d[1] * e2[2] - d[2] * e2[1], d[2] * e2[0] - d[0] * e2[2], d[0] * e2[1] - d[1] * e2[0]};
    const double det = (e1[0] * pv[0] + e1[1] * pv[1]) + e1[2] * pv[2];
    if (!(fabs(det) > 1e-300)) return false;
    const double inv = 1.0 / det;
    const double tv[3] = {o[0] - P0[0], o[1] - P0[1], o[2] - P0[2]};
    u = ((tv[0] * pv[0] + tv[1] * pv[1]) + tv[2] * pv[2]) * inv;
    const double qv[3] = {tv[1] * e1[2] - tv[2] * e1[1], tv[2] * e1[0] - tv[0] * e1[2], tv[0] * e1[1] - tv[1] * e1[0]};
    v = ((qv[0] * d[0] + qv[1] * d[1]) + qv[2] * d[2]) * inv;
    t = ((e2[0] * qv[0] + e2[1] * qv[1]) + e2[2] * qv[2]) * inv;
    return u >= 0.0 && v >= 0.0 && u + v <= 1.0;
}

// Binary32 filter of mt for a crossing parameter in [tmin, tmax]: false only when the
// crossing certainly fails in exact arithmetic by a margin far above the FP64 test's own
// rounding, so mt, run on what passes, decides exactly as without the filter.  Every
// binary32 quantity q below carries an error of at most a few units of 2^-24 times S_q, the
// same expression over the absolute values of its operands: the edge vectors are differences
// of binary32 vertices and round relative to themselves, o - P0 also carries the rounding of o,
// d its own.  The margins are 64 such units.  (Bounding the edges by |P1| + |P0| instead left the
// determinant of a 0.02-wide triangle near the unit sphere undetermined: 35 of the 60 triangles a
// shadow ray met then went on to FP64, against 8 that it crosses.)
// FP64 arithmetic runs at a small fraction of the binary32 rate on this GPU, and most
// boxes the traversal reaches hold triangles the ray misses.
struct RayF {
    dfl o[3], d[3];   // double-float origin and direction; the filter takes the high parts
};
__device__ __forceinline__ dfl df_of(double x) {
    const float h = (float)x;
    return dfl{h, (float)(x - (double)h)};
}
__device__ __forceinline__ double to_double(dfl a) { return (double)a.h + (double)a.l; }
// Error bounds of the filter's determinant and numerators.
struct MtBounds {
    float det, U, V, T;
};
__device__ __forceinline__ bool mt_may_hit(const RayF &r, const float P0[3], const float P1[3], const float P2[3],
                                           float tmin, float tmax, MtBounds &e) {
    constexpr float kU = 64.0f * 0x1p-24f, kTiny = 0x1p-140f;
    float e1[3], e2[3], tv[3], E1[3], E2[3], TV[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        e1[k] = P1[k] - P0[k];
        e2[k] = P2[k] - P0[k];
        tv[k] = r.o[k].h - P0[k];
        E1[k] = fabsf(e1[k]);
        E2[k] = fabsf(e2[k]);
        TV[k] = fabsf(tv[k]) + fabsf(r.o[k].h);
    }
    const float d0 = r.d[0].h, d1 = r.d[1].h, d2 = r.d[2].h;
    const float a0 = fabsf(d0), a1 = fabsf(d1), a2 = fabsf(d2);
    const float pv[3] = {d1 * e2[2] - d2 * e2[1], d2 * e2[0] - d0 * e2[2], d0 * e2[1] - d1 * e2[0]};
    const float PV[3] = {a1 * E2[2] + a2 * E2[1], a2 * E2[0] + a0 * E2[2], a0 * E2[1] + a1 * E2[0]};
    const float det = e1[0] * pv[0] + e1[1] * pv[1] + e1[2] * pv[2];
    // (below 2^-128 the products are rounded in units of 2^-149, above the margins: such triangles go to FP64)
    const float eDet = fmaf(kU, E1[0] * PV[0] + E1[1] * PV[1] + E1[2] * PV[2], 0x1p-128f);
    e = MtBounds{eDet, 3.0e38f, 3.0e38f, 3.0e38f};   // (undetermined: all of it is left to FP64)
    if (!(fabsf(det) > eDet)) return true;
    const float sg = det > 0.0f ? 1.0f : -1.0f;
    const float U = tv[0] * pv[0] + tv[1] * pv[1] + tv[2] * pv[2];
    const float eU = fmaf(kU, TV[0] * PV[0] + TV[1] * PV[1] + TV[2] * PV[2], kTiny);
    if (sg * U < -eU) return false;
    const float qv[3] = {tv[1] * e1[2] - tv[2] * e1[1], tv[2] * e1[0] - tv[0] * e1[2], tv[0] * e1[1] - tv[1] * e1[0]};
    const float QV[3] = {TV[1] * E1[2] + TV[2] * E1[1], TV[2] * E1[0] + TV[0] * E1[2], TV[0] * E1[1] + TV[1] * E1[0]};
    const float V = qv[0] * d0 + qv[1] * d1 + qv[2] * d2;
    const float eV = fmaf(kU, QV[0] * a0 + QV[1] * a1 + QV[2] * a2, kTiny);
    if (sg * V < -eV) return false;
    if (sg * (U + V - det) > eU + eV + eDet) return false;
    const float Tn = e2[0] * qv[0] + e2[1] * qv[1] + e2[2] * qv[2];
    const float eT = fmaf(kU, E2[0] * QV[0] + E2[1] * QV[1] + E2[2] * QV[2], kTiny);
    const float t = Tn / det;
    const float dt = (eT + fabsf(t) * eDet) / (fabsf(det) - eDet) + kU * fabsf(t);
    e = MtBounds{eDet, eU, eV, eT};
    return t + dt >= tmin && t - dt <= tmax;
}

// The same crossing in double-float, whose operations carry errors of at most 2^-42 of the same
// sums: 1 crossing within (tmin, tmax), 0 none, -1 a quantity closer to its limit than 2^-40 of
// the sums (64 units of 2^-24 scaled by 2^-22), which leaves the triangle to the FP64 test.
// FP64's own rounding is far inside the margin, so the decisions are those of the FP64 test.
__device__ __forceinline__ dfl df_det2(dfl a, dfl b, dfl c, dfl d) { return df_add_fast(df_mul(a, b), df_neg(df_mul(c, d))); }
__device__ __forceinline__ dfl df_dot(const dfl a[3], const dfl b[3]) {
    return df_add_fast(df_add_fast(df_mul(a[0], b[0]), df_mul(a[1], b[1])), df_mul(a[2], b[2]));
}
__device__ __forceinline__ int mt_df(const RayF &r, const float P0[3], const float P1[3], const float P2[3],
                                     const MtBounds &e, dfl tmin, dfl tmax, SegHit &h) {
    constexpr float kS = 0x1p-22f;
    const float eD = kS * e.det, eU = kS * e.U, eV = kS * e.V;
    dfl e1[3], e2[3], tv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        e1[k] = df_two_sum(P1[k], -P0[k]);
        e2[k] = df_two_sum(P2[k], -P0[k]);
        tv[k] = df_add_f(r.o[k], -P0[k]);
    }
    const dfl pv[3] = {df_det2(r.d[1], e2[2], r.d[2], e2[1]), df_det2(r.d[2], e2[0], r.d[0], e2[2]),
                       df_det2(r.d[0], e2[1], r.d[1], e2[0])};
    const dfl det = df_dot(e1, pv), U = df_dot(tv, pv);
    // (below 2^-80 the products' low parts could leave binary32's range)
    if (!(fabsf(det.h) > eD && fabsf(U.h) > eU && e.det > 0x1p-80f && e.U < 1.0e38f)) return -1;
    const float sg = det.h > 0.0f ? 1.0f : -1.0f;
    if (sg * U.h < 0.0f) return 0;
    const dfl qv[3] = {df_det2(tv[1], e1[2], tv[2], e1[1]), df_det2(tv[2], e1[0], tv[0], e1[2]),
                       df_det2(tv[0], e1[1], tv[1], e1[0])};
    const dfl V = df_dot(qv, r.d);
    const dfl W = df_add_fast(df_add_fast(U, V), df_neg(det));
    if (!(fabsf(V.h) > eV && fabsf(W.h) > eU + eV + eD)) return -1;
    if (sg * V.h < 0.0f || sg * W.h > 0.0f) return 0;
    h.t = df_div_rcp(df_dot(e2, qv), det);
    const float dt = kS * ((e.T + fabsf(h.t.h) * e.det) / fabsf(det.h)) + 0x1p-40f * fabsf(h.t.h);
    const float below = df_add_fast(h.t, df_neg(tmin)).h, above = df_add_fast(h.t, df_neg(tmax)).h;
    if (!(fabsf(below) > dt && fabsf(above) > dt)) return -1;
    if (below < 0.0f || above > 0.0f) return 0;
    h.u = df_div_rcp(U, det);
    h.v = df_div_rcp(V, det);
    return 1;
}

__device__ __forceinline__ void tri_f(const TraceArgs &a, int tri, float P[3][3]) {
    int64_t v[3];
    tri_verts(a.tris, a.K, tri, v);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int r = 0; r < 3; ++r) P[k][r] = __ldg(a.xyz + 3 * v[k] + r);
}

// The crossing of o + t d with triangle P in FP64.
__device__ __forceinline__ bool crosses_exactly(const double o[3], const double d[3], const float P[3][3], double &t,
                                                double &u, double &v) {
    double Q[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int r = 0; r < 3; ++r) Q[k][r] = (double)P[k][r];
    return mt(o, d, Q[0], Q[1], Q[2], t, u, v);
}
// Whether the segment crosses triangle P inside its ends: the binary32 filter, then double-float, then
// FP64 where neither is certain, from the segment's own FP64 ends (rest: what its double-float origin
// leaves of the FP64 one).
__device__ __forceinline__ bool segment_crosses(const RayF &rf, const float rest[3], const float light[3],
                                                const float P[3][3], SegHit &h) {
    MtBounds e;
    if (!mt_may_hit(rf, P[0], P[1], P[2], (float)kSegEps, (float)(1.0 - kSegEps), e)) return false;
    const int c = mt_df(rf, P[0], P[1], P[2], e, df_of(kSegEps), df_of(1.0 - kSegEps), h);
    if (c >= 0) return c != 0;
    double o[3], d[3], t, u, v;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o[k] = to_double(rf.o[k]) + (double)rest[k];
        d[k] = (double)light[k] - o[k];
    }
    if (!(crosses_exactly(o, d, P, t, u, v) && t > kSegEps && t < 1.0 - kSegEps)) return false;
    h.u = df_of(u);
    h.v = df_of(v);
    return true;
}

// The boxes and children of an internal node.
struct NodeW {
    float4 a, b, c;
    int left, right;
};
__device__ __forceinline__ NodeW load_node(const BvhNode *nodes, int node) {
    const float4 *p = reinterpret_cast<const float4 *>(nodes + node);
    NodeW w;
    w.a = __ldg(p);
    w.b = __ldg(p + 1);
    w.c = __ldg(p + 2);
    const int2 ch = __ldg(reinterpret_cast<const int2 *>(p + 3));
    w.left = ch.x;
    w.right = ch.y;
    return w;
}

// 1 / d, finite: a side that holds the whole ray (0 / 0 otherwise) is then met at t = 0 only, which may
// lose the box but no crossing, as the sides lie at least 16 roundings outside the triangles.
__device__ __forceinline__ float finite_rcp(float d) { return fminf(fmaxf(1.0f / d, -3.0e38f), 3.0e38f); }

// Slab test of the ray o + t d against a box (binary32, widened): whether it meets [t0, t1],
// and where (tn, tf).
__device__ __forceinline__ bool box_span(float lx, float ly, float lz, float hx, float hy, float hz, const float o[3],
                                         const float id[3], float t0, float t1, float &tn, float &tf) {
    const float lo[3] = {lx, ly, lz}, hi[3] = {hx, hy, hz};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float x = (lo[r] - o[r]) * id[r], y = (hi[r] - o[r]) * id[r];
        t0 = fmaxf(t0, fminf(x, y));
        t1 = fminf(t1, fmaxf(x, y));
    }
    tn = t0;
    tf = t1;
    return t0 <= t1;
}
__device__ __forceinline__ bool left_span(const NodeW &w, const float o[3], const float id[3], float t0, float t1,
                                          float &tn, float &tf) {
    return box_span(w.a.x, w.a.y, w.a.z, w.a.w, w.b.x, w.b.y, o, id, t0, t1, tn, tf);
}
__device__ __forceinline__ bool right_span(const NodeW &w, const float o[3], const float id[3], float t0, float t1,
                                           float &tn, float &tf) {
    return box_span(w.b.z, w.b.w, w.c.x, w.c.y, w.c.z, w.c.w, o, id, t0, t1, tn, tf);
}

// Order of crossings. (Their t are positive, and one negative value stands for none: such doubles order like their
// bits, and integer comparisons do not wait for the FP64 unit.)
__device__ __forceinline__ bool hit_less(double ta, int ia, double tb, int ib) {
    const long long a = __double_as_longlong(ta), b = __double_as_longlong(tb);
    return a < b || (a == b && ia < ib);
}
// a0 (1 - u - v) + a1 u + a2 v, in FP64 for the rays and in double-float for the segments.
__device__ __forceinline__ double bary_mix(const double2 uv, float a0, float a1, float a2) {
    return (1.0 - uv.x - uv.y) * a0 + uv.x * a1 + uv.y * a2;
}
__device__ __forceinline__ dfl bary_mix(dfl u, dfl v, float a0, float a1, float a2) {
    const dfl w = df_add_f(df_neg(df_add_fast(u, v)), 1.0f);
    return df_add_fast(df_add_fast(df_mul_f(w, a0), df_mul_f(u, a1)), df_mul_f(v, a2));
}

// A warp's ring of triangles that passed the filter, and what the exact tests made of 32.
struct WarpRing {
    uint2 job[64];            // (lane or segment slot, triangle)
    union {
        double t[32];         // rays: crossings,
        float2 f[32];         // segments: factors of their transmittance
    };
    double u[32], v[32];
    unsigned mine[32];        // rays: per lane of the warp, its crossings among the 32
};
struct Block {
    double d[3][kTracePix];      // the pixels' ray directions
};
static_assert(sizeof(Block) % 16 == 0 && sizeof(WarpRing) % 16 == 0, "shared memory alignment");
// Shadow segments of one block's crossings of one pass, a slot per (crossing, pixel). (31 KB a block: with 33 KB, and
// the smaller L1 that five such blocks leave an SM, the segments take 6% longer.)
constexpr int kJobs = kTraceKB<true> * kTracePix;
struct Jobs {
    float2 o[3][kJobs];                // origin (the segment runs to the light),
    float rest[3][kJobs];              // and its bits below double-float
    float2 S[kJobs];                   // transmittance
    int tri[kJobs];                    // the crossing's own triangle; -1 once the light is blocked to within T_eps
    uint16_t list[kJobs];              // slots in use
    int n, next;
};

// Nodes from here on are leaves; a lane that is not in the tree (node -1) is below it, in an empty scene too.
__device__ __forceinline__ int first_leaf(const TraceArgs &a) { return a.T > 0 ? (int)(a.T - 1) : 0; }

__device__ __forceinline__ void segment(const TraceArgs &a, const Jobs &J, int slot, RayF &rf) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float2 o = J.o[r][slot];
        rf.o[r] = dfl{o.x, o.y};
        rf.d[r] = df_add_f(df_neg(rf.o[r]), a.Lf[r]);
    }
}

// Transmittance of the block's segments through every triangle but their own.  A lane that is done
// takes the next segment of the list, so no lane waits for the longest of 32; what passes the filter (one
// triangle in eight) goes into a ring, and the warp takes 32 of them through the double-float test at
// once (a lane on its own took it with 3 of 32 lanes: 118 -> 46 ms for the 5.4M segments below).
__device__ __forceinline__ void shadow_jobs(const TraceArgs &a, Jobs &J, WarpRing &R) {
    const int n1 = first_leaf(a);
    const float t0 = -1e-3f, t1 = 1.001f;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int stack[kStack];
    int sp = 0, node = -1, slot = 0, own = -1;
    RayF rf;
    float of[3], id[3];
    bool live = true;                // has a segment, or may find one
    uint32_t head = 0, queued = 0;   // the ring
    for (;;) {
        if (live && node < 0) {
            const int j = atomicAdd(&J.next, 1);
            live = j < J.n;
            if (live) {
                slot = J.list[j];
                own = J.tri[slot];
                segment(a, J, slot, rf);
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    of[r] = rf.o[r].h;
                    id[r] = finite_rcp(rf.d[r].h);
                }
                J.S[slot] = make_float2(1.0f, 0.0f);
                sp = 0;
                node = 0;
            }
        }
        // down the tree, until most lanes wait (at a leaf, or for a segment)
        for (;;) {
            const bool inner = node >= 0 && node < n1;
            const unsigned m = __ballot_sync(0xffffffffu, inner), w = __ballot_sync(0xffffffffu, !inner && live);
            if (m == 0 || __popc(m) <= kWalkShare * __popc(w)) break;
            if (inner) {
                const NodeW nd = load_node(a.nodes, node);
                float tn, tf;
                const bool hl = left_span(nd, of, id, t0, t1, tn, tf), hr = right_span(nd, of, id, t0, t1, tn, tf);
                if (hl && hr) {
                    if (sp < kStack) stack[sp++] = nd.right;
                    else atomicAdd(a.overflow, 1u);
                }
                node = hl ? nd.left : (hr ? nd.right : (sp > 0 ? stack[--sp] : -1));
            }
        }
        bool pass = false;
        int tri = -1;
        if (node >= n1) {
            tri = __ldg(a.leaf_tri + (node - n1));
            node = sp > 0 ? stack[--sp] : -1;
            if (tri != own) {
                float P[3][3];
                tri_f(a, tri, P);
                MtBounds e;
                pass = mt_may_hit(rf, P[0], P[1], P[2], (float)kSegEps, (float)(1.0 - kSegEps), e);
            }
        }
        const unsigned c = __ballot_sync(0xffffffffu, pass);
        if (pass) R.job[(head + queued + __popc(c & lt)) & 63u] = make_uint2((uint32_t)slot, (uint32_t)tri);
        queued += __popc(c);
        const bool more = __any_sync(0xffffffffu, live);
        __syncwarp();
        if (queued >= 32u || !more) {
            while (queued >= 32u || (!more && queued)) {
                const uint32_t nj = min(queued, 32u);
                int at = -1;
                if (lane < nj) {
                    const uint2 job = R.job[(head + lane) & 63u];
                    RayF jr;
                    segment(a, J, (int)job.x, jr);
                    float P[3][3];
                    tri_f(a, (int)job.y, P);
                    SegHit h;
                    const float rest[3] = {J.rest[0][job.x], J.rest[1][job.x], J.rest[2][job.x]};
                    if (segment_crosses(jr, rest, a.Lf, P, h)) {
                        int64_t v[3];
                        tri_verts(a.tris, a.K, (int)job.y, v);
                        const dfl al = bary_mix(h.u, h.v, __ldg(a.alpha + v[0]), __ldg(a.alpha + v[1]), __ldg(a.alpha + v[2]));
                        const dfl f = df_add_f(df_neg(al), 1.0f);
                        R.f[lane] = make_float2(f.h, f.l);
                        at = (int)job.x;
                    }
                }
                head += nj;
                queued -= nj;
                // a segment's factors in the order it met them, by the first of their lanes, up to the one
                // that blocks the light to within T_eps: the colour's shadow factor moves by at most
                // (1 - ambient) T_eps, the primary composite's own termination bound (what comes after
                // is left out whenever it is tested, so the product does not depend on the warp's other
                // segments)
                unsigned same = __match_any_sync(0xffffffffu, at);
                __syncwarp();
                if (at >= 0 && lane == __ffs(same) - 1 && J.tri[at] >= 0) {
                    dfl S = dfl{J.S[at].x, J.S[at].y};
                    for (; same; same &= same - 1) {
                        const float2 f = R.f[__ffs(same) - 1];
                        S = df_mul(S, dfl{f.x, f.y});
                        if (df_lt(S, df_make(a.T_epsf))) {
                            J.tri[at] = -1;
                            break;
                        }
                    }
                    J.S[at] = make_float2(S.h, S.l);
                }
                __syncwarp();
            }
            if (node >= 0 && J.tri[slot] < 0) node = -1;   // (the lane's own segment: it takes the next)
        }
        if (!more) break;
    }
}

// One lane a pixel, a warp 8 x 4 pixels, so that its rays stay together down the tree.  With shadows a
// block is one such warp and three more: it gathers its pixels' next crossings, all four trace
// their segments to the light as one list, and it composites.  What bounds it: the waits on nodes, lanes at
// different depths of the tree (18 of 32 active; a segment meets 187 nodes and 60 leaves), and the blocks with
// the deepest pixels at the end.  1.6M triangles at 800x800: 5.1 ms without shadows, 39 ms with the 5.4M
// segments; 41 and 148 ms for lanes that each took their triangles through the exact tests alone
// (4.5 of 32 active); 62 ms with two warps for 8 x 8 pixels and their segments, whose deepest blocks left
// two thirds of the chip idle; 218 ms for a thread that traced its own pixel's segments one after the other.
template <bool SHADOWS>
__global__ void __launch_bounds__(32 * (SHADOWS ? kTraceWarps : kPlainWarps), SHADOWS ? kTraceBlocks : 0)
trace_kernel(const __grid_constant__ TraceArgs a) {
    extern __shared__ __align__(16) char smem[];
    // a ring for each warp, the block's words, and with shadows its segments
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpRing &R = reinterpret_cast<WarpRing *>(smem)[warp];
    char *rest = smem + (SHADOWS ? kTraceWarps : kPlainWarps) * sizeof(WarpRing);
    Block &B = reinterpret_cast<Block *>(rest)[SHADOWS ? 0 : warp];
    Jobs &J = *reinterpret_cast<Jobs *>(rest + sizeof(Block));
    const bool lead = !SHADOWS || warp == 0;   // a warp of pixels
    const unsigned lt = (1u << lane) - 1u;
    const int W = a.cam.width, H = a.cam.height;
    const int px = blockIdx.x * 8 + (lane & 7), py = blockIdx.y * (SHADOWS ? 4 : 4 * kPlainWarps) + (SHADOWS ? 0 : 4 * warp) + (lane >> 3);
    const bool in = lead && px < W && py < H;
    const CamDev &c = a.cam;
    RayF rf;
    float of[3], id[3];
    {
        // ray with unit view depth: d = R^T ((x - cx) / fx, (y - cy) / fy, 1)
        const double dc[3] = {((double)px + 0.5 - (double)c.cx) / (double)c.fx,
                              ((double)py + 0.5 - (double)c.cy) / (double)c.fy, 1.0};
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            rf.o[r] = df_make(c.C[r]);
            const double d = ((double)c.R[r] * dc[0] + (double)c.R[3 + r] * dc[1]) + (double)c.R[6 + r] * dc[2];
            rf.d[r] = df_of(d);
            of[r] = rf.o[r].h;
            id[r] = finite_rcp(rf.d[r].h);
            if (lead) B.d[r][lane] = d;
        }
    }
    const int n1 = first_leaf(a);
    double T = 1.0, C0 = 0.0, C1 = 0.0, C2 = 0.0;
    double after_t = -1.0e300;
    int after_i = -1;
    bool alive = in && a.T > 0;
    for (;;) {
        Hit buf[kTraceKB<SHADOWS>];
        double2 uv[kTraceKB<SHADOWS>];
        int nb = 0;
        bool more = false;
        int n_use = 0;
        if (lead) {
            // The warp's pixels walk the tree together, as the segments do (shadow_jobs): triangles that
            // pass the filter wait in the ring for the FP64 test of 32, and each lane sorts its own
            // crossings of these into its buffer.
            int stack[kStack];
            int sp = 0, node = alive ? 0 : -1;
            uint32_t head = 0, queued = 0;
            // Boxes wholly before the last composited crossing hold nothing for this pass, and
            // boxes wholly beyond the farthest kept crossing of a full buffer only mean another
            // pass; both bounds are widened by 1e-5 relative, far above the slab test's rounding.
            const float after_f = fmaxf((float)after_t, 0.0f), t_after = after_f * (1.0f - 1e-5f);
            const float t_near = c.znear * 0.999f;
            for (;;) {
                for (;;) {
                    const bool inner = node >= 0 && node < n1;
                    const unsigned m = __ballot_sync(0xffffffffu, inner), w = __ballot_sync(0xffffffffu, node >= n1);
                    if (m == 0 || __popc(m) <= kWalkShare * __popc(w)) break;
                    if (!inner) continue;
                    const NodeW nd = load_node(a.nodes, node);
                    float nl, fl, nr, fr;
                    bool hl = left_span(nd, of, id, t_near, 3.0e38f, nl, fl) && fl >= t_after;
                    bool hr = right_span(nd, of, id, t_near, 3.0e38f, nr, fr) && fr >= t_after;
                    if (nb == kTraceKB<SHADOWS>) {
                        const float t_far = (float)buf[kTraceKB<SHADOWS> - 1].t * (1.0f + 1e-5f);
                        if (hl && nl > t_far) {
                            hl = false;
                            more = true;
                        }
                        if (hr && nr > t_far) {
                            hr = false;
                            more = true;
                        }
                    }
                    // the nearer child first: the buffer fills with near crossings early
                    const bool swap = hl && hr && nr < nl;
                    const int first = swap || !hl ? nd.right : nd.left, second = swap ? nd.left : nd.right;
                    if (hl && hr) {
                        if (sp < kStack) stack[sp++] = second;
                        else atomicAdd(a.overflow, 1u);
                    }
                    node = hl || hr ? first : (sp > 0 ? stack[--sp] : -1);
                }
                bool pass = false;
                int tri = -1;
                if (node >= n1) {
                    tri = __ldg(a.leaf_tri + (node - n1));
                    node = sp > 0 ? stack[--sp] : -1;
                    float P[3][3];
                    tri_f(a, tri, P);
                    MtBounds e;
                    // (crossings before the last composited one were taken in an earlier pass)
                    pass = mt_may_hit(rf, P[0], P[1], P[2], fmaxf(c.znear, after_f), 3.0e38f, e);
                }
                const unsigned cand = __ballot_sync(0xffffffffu, pass);
                if (pass) R.job[(head + queued + __popc(cand & lt)) & 63u] = make_uint2((uint32_t)lane, (uint32_t)tri);
                queued += __popc(cand);
                const bool walking = __any_sync(0xffffffffu, node >= 0);
                __syncwarp();
                while (queued >= 32u || (!walking && queued)) {
                    const uint32_t nj = min(queued, 32u);
                    int owner = -1;
                    if (lane < nj) {
                        const uint2 job = R.job[(head + lane) & 63u];
                        const int at = (int)job.x;
                        double o[3], d[3], t, u, v;
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
                            o[r] = (double)c.C[r];
                            d[r] = B.d[r][at];
                        }
                        float P[3][3];
                        tri_f(a, (int)job.y, P);
                        if (crosses_exactly(o, d, P, t, u, v) && t > (double)c.znear) {
                            owner = at;
                            R.t[lane] = t;
                            R.u[lane] = u;
                            R.v[lane] = v;
                        }
                    }
                    R.mine[lane] = 0;
                    const unsigned same = __match_any_sync(0xffffffffu, owner);
                    __syncwarp();
                    if (owner >= 0 && lane == __ffs(same) - 1) R.mine[owner] = same;
                    __syncwarp();
                    for (unsigned b = R.mine[lane]; b; b &= b - 1) {
                        const int i = __ffs(b) - 1;
                        Hit h = {R.t[i], (int)R.job[(head + i) & 63u].y, nb};
                        if (!hit_less(after_t, after_i, h.t, h.tri)) continue;   // composited in an earlier pass
                        if (nb == kTraceKB<SHADOWS>) {
                            more = true;
                            if (!hit_less(h.t, h.tri, buf[kTraceKB<SHADOWS> - 1].t, buf[kTraceKB<SHADOWS> - 1].tri)) continue;
                            --nb;   // the farthest kept crossing waits for a later pass
                            h.at = buf[nb].at;
                        }
                        int s = nb;
                        while (s > 0 && hit_less(h.t, h.tri, buf[s - 1].t, buf[s - 1].tri)) {
                            buf[s] = buf[s - 1];
                            --s;
                        }
                        buf[s] = h;
                        uv[h.at] = make_double2(R.u[i], R.v[i]);
                        ++nb;
                    }
                    __syncwarp();
                    head += nj;
                    queued -= nj;
                }
                if (!walking) break;
            }
            // the crossings that will be composited: up to the one that takes T below T_eps (known once they are
            // composited, where there are no segments to trace first)
            n_use = nb;
            if (SHADOWS) {
                double Tn = T;
                n_use = 0;
                for (bool on = true; on && n_use < nb; ++n_use, on = !(Tn < a.T_eps)) {
                    const Hit &h = buf[n_use];
                    int64_t v[3];
                    tri_verts(a.tris, a.K, h.tri, v);
                    Tn *= 1.0 - bary_mix(uv[h.at], __ldg(a.alpha + v[0]), __ldg(a.alpha + v[1]), __ldg(a.alpha + v[2]));
                }
            }
        }
        if (SHADOWS) {
            if (lead) {
                int n = 0;
                for (int k = 0; k < kTraceKB<SHADOWS>; ++k) {   // the segments of one depth follow each other
                    const bool has = k < n_use;
                    const unsigned m = __ballot_sync(0xffffffffu, has);
                    if (has) {
                        const int slot = k * kTracePix + lane;
                        J.list[n + __popc(m & lt)] = (uint16_t)slot;
                        J.tri[slot] = buf[k].tri;
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
                            const double p = (double)c.C[r] + buf[k].t * B.d[r][lane];
                            const dfl pf = df_of(p);
                            J.o[r][slot] = make_float2(pf.h, pf.l);
                            J.rest[r][slot] = (float)(p - to_double(pf));
                        }
                    }
                    n += __popc(m);
                }
                if (lane == 0) {
                    J.n = n;
                    J.next = 0;
                }
            }
            __syncthreads();
            shadow_jobs(a, J, R);
            __syncthreads();
        }
        for (int k = 0; k < n_use; ++k) {
            const Hit &h = buf[k];
            const double2 q = uv[h.at];
            int64_t v[3];
            tri_verts(a.tris, a.K, h.tri, v);
            const double al = bary_mix(q, __ldg(a.alpha + v[0]), __ldg(a.alpha + v[1]), __ldg(a.alpha + v[2]));
            double col[3];
#pragma unroll
            for (int r = 0; r < 3; ++r)
                col[r] = bary_mix(q, __ldg(a.rgb + 3 * v[0] + r), __ldg(a.rgb + 3 * v[1] + r), __ldg(a.rgb + 3 * v[2] + r));
            if (SHADOWS) {
                const float2 S = J.S[k * kTracePix + lane];
                const double f = a.ambient + (1.0 - a.ambient) * to_double(dfl{S.x, S.y});
#pragma unroll
                for (int r = 0; r < 3; ++r) col[r] *= f;
            }
            C0 += T * al * col[0];
            C1 += T * al * col[1];
            C2 += T * al * col[2];
            T *= 1.0 - al;
            after_t = h.t;
            after_i = h.tri;
            if (!SHADOWS && T < a.T_eps) break;
        }
        alive = alive && more && !(T < a.T_eps);
        if (SHADOWS ? !__syncthreads_or(alive) : !__any_sync(0xffffffffu, alive)) break;
    }
    if (!in) return;
    float4 *out = reinterpret_cast<float4 *>(a.out);
    out[(int64_t)py * W + px] = make_float4((float)(C0 + T * a.bg[0]), (float)(C1 + T * a.bg[1]),
                                            (float)(C2 + T * a.bg[2]), (float)(1.0 - T));
}

unsigned grid_of(int64_t n, int threads) {
    return (unsigned)min64((n + threads - 1) / threads, (int64_t)32 * 152);
}

}  // namespace
}  // namespace ms

using namespace ms;

extern "C" MS_API size_t ms_bvh_workspace_size(int64_t T) {
    if (T < 0) return 0;
    return bvh_layout(T).total;
}

extern "C" MS_API ms_status ms_bvh_build(const float *xyz, const int32_t *tris, int64_t T, int32_t K, void *bvh,
                                         size_t bvh_bytes, void *stream) {
    if (T < 0 || T >= (1ll << 31)) return set_error(MS_ERR_INVALID, "T outside 0 .. 2^31 - 1");
    if (!tris && (K < 3 || K > kMaxK || T % K)) return set_error(MS_ERR_INVALID, "implicit fans need K in 3..16 and T % K == 0");
    if (T > 0 && !xyz) return set_error(MS_ERR_INVALID, "xyz is NULL");
    const BvhLayout L = bvh_layout(T);
    if (!bvh || (reinterpret_cast<uintptr_t>(bvh) & 255) || bvh_bytes < L.total)
        return set_error(MS_ERR_INVALID, "BVH workspace NULL, misaligned or < %zu bytes", L.total);
    cudaStream_t st = (cudaStream_t)stream;
    char *b = static_cast<char *>(bvh);
    cudaError_t e = cudaMemsetAsync(b, 0, L.nodes, st);   // status and bounds
    if (e == cudaSuccess && T > 0) e = cudaMemsetAsync(b + L.flags, 0, (size_t)T * 4, st);
    if (e != cudaSuccess) return set_error(MS_ERR_CUDA, "memset: %s", cudaGetErrorString(e));
    if (T == 0) return MS_OK;
    unsigned *bounds = reinterpret_cast<unsigned *>(b + L.bounds);
    bounds_init_kernel<<<1, 32, 0, st>>>(bounds);
    centroid_bounds_kernel<<<grid_of(T, kBvhThreads), kBvhThreads, 0, st>>>(xyz, tris, K, T, bounds);
    unsigned long long *k0 = reinterpret_cast<unsigned long long *>(b + L.keys0);
    unsigned long long *k1 = reinterpret_cast<unsigned long long *>(b + L.keys1);
    morton_kernel<<<grid_of(T, kBvhThreads), kBvhThreads, 0, st>>>(xyz, tris, K, T, bounds, k0);
    unsigned long long *sorted = k0;
    e = sort_u64(k0, k1, T, 32, 4, b + L.scratch, st, &sorted);
    if (e != cudaSuccess) return set_error(MS_ERR_CUDA, "BVH key sort: %s", cudaGetErrorString(e));
    BvhNode *nodes = reinterpret_cast<BvhNode *>(b + L.nodes);
    uint32_t *parent = reinterpret_cast<uint32_t *>(b + L.parent);
    int *leaf_tri = reinterpret_cast<int *>(b + L.leaf_tri);
    radix_tree_kernel<<<grid_of(T, kBvhThreads), kBvhThreads, 0, st>>>(sorted, T, nodes, parent, leaf_tri);
    bounds_up_kernel<<<grid_of(T, kBvhThreads), kBvhThreads, 0, st>>>(xyz, tris, K, T, nodes, parent, leaf_tri,
                                                                      reinterpret_cast<int *>(b + L.flags));
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(MS_ERR_CUDA, "BVH build: %s", cudaGetErrorString(e));
    count_launches(5);
    return MS_OK;
}

extern "C" MS_API ms_status ms_raytrace(const float *xyz, const float *rgb, const float *alpha, const int32_t *tris,
                                        int64_t T, int32_t K, const void *bvh, const ms_camera *cam,
                                        const float *light, float ambient, float T_eps, const float *bg,
                                        float *out_rgba, void *stream) {
    if (T < 0 || T >= (1ll << 31)) return set_error(MS_ERR_INVALID, "T outside 0 .. 2^31 - 1");
    if (!tris && (K < 3 || K > kMaxK || T % K)) return set_error(MS_ERR_INVALID, "implicit fans need K in 3..16 and T % K == 0");
    if (!cam || !out_rgba || (T > 0 && (!xyz || !rgb || !alpha || !bvh)))
        return set_error(MS_ERR_INVALID, "NULL pointer");
    if (cam->width <= 0 || cam->height <= 0 || cam->width > 32768 || cam->height > 32768 || !(cam->znear > 0.0f))
        return set_error(MS_ERR_INVALID, "camera");
    if (!(ambient >= 0.0f && ambient <= 1.0f)) return set_error(MS_ERR_INVALID, "ambient outside [0, 1]");
    if (reinterpret_cast<uintptr_t>(out_rgba) & 15) return set_error(MS_ERR_INVALID, "out_rgba not 16-byte aligned");
    const BvhLayout L = bvh_layout(T);
    TraceArgs a;
    a.xyz = xyz;
    a.rgb = rgb;
    a.alpha = alpha;
    a.tris = tris;
    a.K = K;
    a.T = T;
    const char *b = static_cast<const char *>(bvh);
    a.nodes = T > 0 ? reinterpret_cast<const BvhNode *>(b + L.nodes) : nullptr;
    a.leaf_tri = T > 0 ? reinterpret_cast<const int *>(b + L.leaf_tri) : nullptr;
    a.overflow = T > 0 ? reinterpret_cast<unsigned *>(const_cast<char *>(b) + L.status) : nullptr;
    a.cam = make_cam(*cam);
    a.shadows = light != nullptr && ambient < 1.0f;
    for (int r = 0; r < 3; ++r) {
        a.Lf[r] = light ? light[r] : 0.0f;
        a.bg[r] = bg ? bg[r] : 0.0f;
    }
    a.ambient = ambient;
    a.T_eps = a.T_epsf = T_eps;
    a.out = out_rgba;
    const int rows = a.shadows ? 4 : 4 * kPlainWarps;
    const dim3 grid((cam->width + 7) / 8, (cam->height + rows - 1) / rows);
    if (a.shadows)
        trace_kernel<true><<<grid, 32 * kTraceWarps, kTraceWarps * sizeof(WarpRing) + sizeof(Block) + sizeof(Jobs), (cudaStream_t)stream>>>(a);
    else
        trace_kernel<false><<<grid, 32 * kPlainWarps, kPlainWarps * (sizeof(WarpRing) + sizeof(Block)), (cudaStream_t)stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(MS_ERR_CUDA, "trace_kernel: %s", cudaGetErrorString(e));
    count_launches(1);
    return MS_OK;
}

extern "C" MS_API ms_status ms_bvh_status(const void *bvh, int32_t *stack_overflows, void *stream) {
    if (!bvh || !stack_overflows) return set_error(MS_ERR_INVALID, "NULL pointer");
    unsigned v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, bvh, sizeof(unsigned), cudaMemcpyDeviceToHost, (cudaStream_t)stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess) return set_error(MS_ERR_CUDA, "status read: %s", cudaGetErrorString(e));
    *stack_overflows = (int32_t)v;
    return v ? MS_ERR_CAPACITY : MS_OK;
}
