// Gaussian -> triangle-fan conversion with SH colour (Sec. 3, "MeshSplats
// Transformation for Flat Gaussians", Eq. 2 and the vertex equation after it; and
// "Transformation for 3D Gaussians": all three scaled axes kept, one fan per pair of axes
// (1, 2), (1, 3), (2, 3), written as three implicit fans of K triangles per Gaussian whose
// shared vertices -- the centre and the axis tips two fans reach -- are copies; the
// angle table then holds exact cosine and sine at quarter turns, so the copies are equal
// bit for bit).
//
// One thread per Gaussian forms its frame (mb::gaussian_frame: centre, scaled axes, colour,
// opacity) in shared memory, 13 or 16 floats; the block's threads then form the output words
// where they are stored, four consecutive words of an array each.  Read 44 B + SH, write
// 28 (K+1) B per fan, bound by those bytes; a frame in place of the staged vertices (7 (K+1) floats
// a fan) lets the threads, not the shared memory, limit the blocks per SM.  1M
// Gaussians (bf16 SH degree 3, K = 8): 92.4 -> 77.9 us a call; 200k into three fans (f32 SH):
// 60.7 -> 52.3 us.
// With given corrections every vertex has its own, and a thread stages its Gaussian's vertices.
#include "mesh_build.cuh"

namespace ms {

namespace {

constexpr int kMBThreads = 128;

// Rows of a frame in shared memory: centre, axes, colour, opacity (an odd length spreads the rows
// over the banks; 16 + 1 for three axes).
template <bool THREE>
constexpr int kFrameRow = THREE ? 17 : 13;

// Word r of boundary or centre vertex k (of GV, fan by fan) of the Gaussian with frame f.
template <bool THREE>
__device__ __forceinline__ float xyz_word(const float *f, const float *cs, const float *sn, int KV, int k, int r) {
    int fa = 0, fb = 1;
    if (THREE) {
        const int fan = k >= 2 * KV ? 2 : (k >= KV ? 1 : 0);
        k -= fan * KV;
        fa = fan == 2 ? 1 : 0;
        fb = fan == 0 ? 1 : 2;
    }
    return k == 0 ? f[r] : f[r] + (cs[k - 1] * f[3 + 3 * fa + r] + sn[k - 1] * f[3 + 3 * fb + r]);
}

// Stores n words of dst, word i = value(i / per, i % per) (per words a Gaussian), four at a time
// where dst is aligned.  (i + 0.5) / per is at least 1 / (2 per) away from an integer, far above the
// rounding of i < kMBThreads * 3 * 51.
template <typename F>
__device__ __forceinline__ void store_words(float *__restrict__ dst, int n, int per, F value) {
    const float inv = 1.0f / (float)per;
    if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
        for (int i = 4 * threadIdx.x; i + 4 <= n; i += 4 * kMBThreads) {
            int g = (int)(((float)i + 0.5f) * inv), w = i - g * per;
            float v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q] = value(g, w);
                if (++w == per) {
                    w = 0;
                    ++g;
                }
            }
            *reinterpret_cast<float4 *>(dst + i) = make_float4(v[0], v[1], v[2], v[3]);
        }
        const int i = (n & ~3) + threadIdx.x;
        if (i < n) dst[i] = value(i / per, i % per);
    } else {
        for (int i = threadIdx.x; i < n; i += kMBThreads) {
            const int g = (int)(((float)i + 0.5f) * inv);
            dst[i] = value(g, i - g * per);
        }
    }
}

template <int DEG, bool BF16, bool THREE>
__global__ void __launch_bounds__(kMBThreads) mesh_build_kernel(const mb::Gaussians G, int64_t N,
                                                                const __grid_constant__ MeshBuildConst kc,
                                                                float *__restrict__ xyz, float *__restrict__ rgb,
                                                                float *__restrict__ alpha) {
    constexpr int ROW = kFrameRow<THREE>, COL = THREE ? 12 : 9;
    __shared__ float s_f[kMBThreads * ROW], s_cs[kMaxK], s_sn[kMaxK];
    const int KV = kc.K + 1, GV = (THREE ? 3 : 1) * KV;   // vertices per fan, per Gaussian
    const int64_t g0 = (int64_t)blockIdx.x * kMBThreads, g = g0 + threadIdx.x;
    const int nloc = (int)min64(kMBThreads, N - g0);
    if (threadIdx.x < kMaxK) {
        s_cs[threadIdx.x] = kc.cs[threadIdx.x];
        s_sn[threadIdx.x] = kc.sn[threadIdx.x];
    }
    if (g < N) {
        const mb::Frame F = mb::gaussian_frame<DEG, BF16, THREE>(G, kc, g);
        float *f = s_f + threadIdx.x * ROW;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            f[r] = F.m[r];
            f[3 + r] = F.ax[0][r];
            f[6 + r] = F.ax[1][r];
            if (THREE) f[9 + r] = F.ax[2][r];
            f[COL + r] = F.col[r];
        }
        f[COL + 3] = F.sig;
    }
    __syncthreads();
    const int64_t v0 = g0 * GV;
    store_words(xyz + 3 * v0, 3 * nloc * GV, 3 * GV, [&](int l, int w) {
        const int k = (int)__umulhi((unsigned)w, 0x55555556u);   // w / 3
        return xyz_word<THREE>(s_f + l * ROW, s_cs, s_sn, KV, k, w - 3 * k);
    });
    store_words(rgb + 3 * v0, 3 * nloc * GV, 3 * GV, [&](int l, int w) {
        return s_f[l * ROW + COL + (w - 3 * (int)__umulhi((unsigned)w, 0x55555556u))];
    });
    store_words(alpha + v0, nloc * GV, GV, [&](int l, int w) {
        const float sig = s_f[l * ROW + COL + 3];
        const bool centre = w == 0 || (THREE && (w == KV || w == 2 * KV));
        return centre ? sig : kc.opac_mul * sig;
    });
}

// The conversion with given corrections: a thread stages its Gaussian's vertices.
template <int DEG, bool BF16>
__global__ void __launch_bounds__(kMBThreads) mesh_build_corr_kernel(const mb::Gaussians G, int64_t N, MeshBuildConst kc,
                                                                     const float *__restrict__ corr,
                                                                     float *__restrict__ xyz, float *__restrict__ rgb,
                                                                     float *__restrict__ alpha) {
    extern __shared__ float smem[];
    const int KV = kc.K + 1;
    float *s_xyz = smem;                          // kMBThreads * KV * 3
    float *s_rgb = s_xyz + kMBThreads * KV * 3;   // kMBThreads * KV * 3
    float *s_a = s_rgb + kMBThreads * KV * 3;     // kMBThreads * KV

    const int64_t g0 = (int64_t)blockIdx.x * kMBThreads;
    const int64_t g = g0 + threadIdx.x;
    const int nloc = (int)min64(kMBThreads, N - g0);
    if (g < N)
        mb::convert_gaussian<DEG, BF16>(G, kc, g, corr + g * 2 * KV, s_xyz, s_rgb, s_a, threadIdx.x * KV);
    __syncthreads();
    const int64_t v0 = g0 * KV;
    mb::block_store(xyz + 3 * v0, s_xyz, 3 * nloc * KV);
    mb::block_store(rgb + 3 * v0, s_rgb, 3 * nloc * KV);
    mb::block_store(alpha + v0, s_a, nloc * KV);
}

template <int DEG, bool BF16>
cudaError_t launch_t(const mb::Gaussians &G, int64_t N, const MeshBuildConst &kc, const float *corr, float *xyz,
                     float *rgb, float *alpha, cudaStream_t st) {
    const unsigned grid = (unsigned)((N + kMBThreads - 1) / kMBThreads);
    if (corr && !kc.three) {
        const size_t smem = sizeof(float) * kMBThreads * (kc.K + 1) * 7;
        auto fn = mesh_build_corr_kernel<DEG, BF16>;
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        fn<<<grid, kMBThreads, smem, st>>>(G, N, kc, corr, xyz, rgb, alpha);
    } else if (kc.three) {
        mesh_build_kernel<DEG, BF16, true><<<grid, kMBThreads, 0, st>>>(G, N, kc, xyz, rgb, alpha);
    } else {
        mesh_build_kernel<DEG, BF16, false><<<grid, kMBThreads, 0, st>>>(G, N, kc, xyz, rgb, alpha);
    }
    return cudaGetLastError();
}

template <int DEG>
cudaError_t launch_deg(bool bf16, const float *means, const float *log_scales, const float *quats,
                       const float *opacity, const void *sh, int64_t N, const MeshBuildConst &kc, const float *corr,
                       float *xyz, float *rgb, float *alpha, cudaStream_t st) {
    const mb::Gaussians G{means, log_scales, quats, opacity, sh};
    return bf16 ? launch_t<DEG, true>(G, N, kc, corr, xyz, rgb, alpha, st)
                : launch_t<DEG, false>(G, N, kc, corr, xyz, rgb, alpha, st);
}

}  // namespace

cudaError_t launch_mesh_build(const float *means, const float *log_scales, const float *quats, const float *opacity,
                              const void *sh, int sh_dtype, int sh_degree, int64_t N, const MeshBuildConst &kc,
                              const float *corr, float *xyz, float *rgb, float *alpha, cudaStream_t st) {
    if (N == 0) return cudaSuccess;
    const bool bf16 = sh_dtype == 1;
    switch (sh_degree) {
        case 0: return launch_deg<0>(bf16, means, log_scales, quats, opacity, sh, N, kc, corr, xyz, rgb, alpha, st);
        case 1: return launch_deg<1>(bf16, means, log_scales, quats, opacity, sh, N, kc, corr, xyz, rgb, alpha, st);
        case 2: return launch_deg<2>(bf16, means, log_scales, quats, opacity, sh, N, kc, corr, xyz, rgb, alpha, st);
        default: return launch_deg<3>(bf16, means, log_scales, quats, opacity, sh, N, kc, corr, xyz, rgb, alpha, st);
    }
}

}  // namespace ms
