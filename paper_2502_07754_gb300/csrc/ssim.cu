// Fine-tuning loss of Sec. 3 (Eq. 3), read as lambda L1 + (1 - lambda)(1 - SSIM): SSIM
// per colour channel under an 11 x 11 Gaussian window (sigma 1.5, zero padding outside
// the image, C1 = 0.01^2, C2 = 0.03^2) averaged over the pixels and the three channels.
//
// Two launches, over 32 x 16 (forward) and 32 x 32 output tiles, each staging a window of its inputs five
// pixels wider on each side in shared memory (the forward stages the three channels of image and
// target in one pass) and applying the separable window as a row pass then a column pass.  A thread takes eight
// neighbouring outputs of the row pass and four of the column pass, so a staged value is loaded
// once for the up to eleven products it enters, and the sums go two at a time through packed f32x2
// multiply-adds.  At 1080p the two launches take
// 0.084 + 0.080 ms, against 0.157 + 0.161 ms with one output a thread on 16 x 16 tiles (273 shared loads
// a pixel); issue slots bound them, at 26% of the HBM bandwidth.
//
// ssim_fwd_kernel: per channel the raw local moments (x, y, x^2, y^2, xy), the SSIM map,
//   and the three per-pixel factors of its gradient (with A = 2 mu_x mu_y + C1,
//   B = 2 s_xy + C2, C = mu_x^2 + mu_y^2 + C1, D = s_xx + s_yy + C2, S = AB/(CD)):
//     G2 = dS/ds_xx = -S/D,  G3 = dS/ds_xy = 2A/(CD),
//     G1 = dS/dmu_x - 2 mu_x G2 - mu_y G3,  dS/dmu_x = 2 mu_y B/(CD) - 2 mu_x S/C,
//   written as nine planes; the block's share of the loss is added to *loss.  The
//   moments are taken of x - r_x and y - r_y with one reference value per 16 x 16 square (a pixel
//   near its centre; outside the image the padded zeros become -r; one value for 32 x 32 pixels, as forward tiles of
//   that size had, nearly doubled the gradient's error on steep smooth images, for the same time): the local
//   (co)variances do not depend on the shift, and E[x^2] - mu^2 then cancels against the
//   local contrast instead of against the brightness.
// ssim_bwd_kernel: dSSIM/dx_p = (1/N) [(w * G1)(p) + 2 x_p (w * G2)(p) + y_p (w * G3)(p)],
//   w * G the window sum of a plane over the image's pixels (zero outside), and
//   dL/dx = lambda sign(x - y)/N - (1 - lambda) dSSIM/dx, N = 3 H W.
#include <cmath>

#include "ms_internal.h"

namespace ms {

namespace {

constexpr int kT = 32;                   // output tile edge
constexpr int kR = 5;                    // window radius
constexpr int kIn = kT + 2 * kR;         // staged tile edge (42)
constexpr int kThreads = 256;
constexpr int kRow = 8, kCol = kT * kT / kThreads;   // outputs of a thread in the row and column pass
constexpr int kRowTasks = kIn * (kT / kRow);
// The forward takes 32 x 16 outputs, two 16 x 16 squares with a reference value each.
constexpr int kFH = 16, kFIn = kFH + 2 * kR, kFThreads = 128;
constexpr int kFRowTasks = kFIn * (kT / kRow);
static_assert(kT * kFH / kFThreads == kCol && kFRowTasks <= kFThreads, "forward tile");
constexpr float kC1 = 0.0001f, kC2 = 0.0009f;

struct Window {
    float w[2 * kR + 1];
};

__device__ __forceinline__ float chan(const float4 &v, int c) { return c == 0 ? v.x : (c == 1 ? v.y : v.z); }

// Pairs of binary32 values and their packed multiply and multiply-add (rounded like the scalar ones).
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)),
          "l"(reinterpret_cast<const unsigned long long &>(c)));
    return d;
}

template <int THREADS>
__device__ __forceinline__ float block_sum(float v, float *s_red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int tid = threadIdx.x;
    if ((tid & 31) == 0) s_red[tid >> 5] = v;
    __syncthreads();
    float t = 0.0f;
    if (tid < 32) {
        t = tid < THREADS / 32 ? s_red[tid] : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    return t;
}

// (rows are consecutive over the lanes of the row pass, columns over those of the column pass: the
// odd row lengths keep both free of bank conflicts)
struct FwdMem {
    float2 in[3][kFIn][kIn + 1];     // (x, y) of a channel
    float2 h01[kFIn][kT + 1];        // row sums of x and y, about the square's reference,
    float2 h23[kFIn][kT + 1];        // of x^2 and y^2,
    float h4[kFIn][kT + 1];          // and of x y
    float2 ref[2][3];                // each square's reference (x, y) of a channel
    float red[kFThreads / 32];
};

// The loss over the blocks, summed in FP64: thousands of binary32 additions to one word would
// carry an error of about 1e-6 of it, different from run to run.  The last block rounds it.
struct LossSum {
    double sum;
    unsigned done, pad;
};

__global__ void __launch_bounds__(kFThreads, 5) ssim_fwd_kernel(const float4 *__restrict__ img, const float4 *__restrict__ tgt,
                                                            int H, int W, float lam, float inv_n, Window win,
                                                            float *__restrict__ G, LossSum *total,
                                                            float *__restrict__ loss) {
    __shared__ FwdMem S;
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * kT, y0 = blockIdx.y * kFH;
    const size_t plane = (size_t)H * W;
    float acc = 0.0f;
    if (tid < 2) {
        const size_t ref = (size_t)min(y0 + kFH / 2, H - 1) * W + min(x0 + kFH / 2 + kFH * tid, W - 1);
        const float4 rx = img[ref], ry = tgt[ref];
#pragma unroll
        for (int c = 0; c < 3; ++c) S.ref[tid][c] = make_float2(chan(rx, c), chan(ry, c));
    }
    // one pass over the window stages all three channels (each RGBA pixel loaded once)
    for (int i = tid; i < kFIn * kIn; i += kFThreads) {
        const int ly = i / kIn, lx = i - ly * kIn;
        const int gx = x0 - kR + lx, gy = y0 - kR + ly;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (gx >= 0 && gx < W && gy >= 0 && gy < H) {
            a = img[(size_t)gy * W + gx];
            b = tgt[(size_t)gy * W + gx];
            if (lx >= kR && lx < kR + kT && ly >= kR && ly < kR + kFH)
                acc += lam * (fabsf(a.x - b.x) + fabsf(a.y - b.y) + fabsf(a.z - b.z));
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) S.in[c][ly][lx] = make_float2(chan(a, c), chan(b, c));
    }
    __syncthreads();
    const int tx = tid & 31, ty = (tid >> 5) * kCol;
    const int px = x0 + tx;
    for (int c = 0; c < 3; ++c) {
        if (tid < kFRowTasks) {
            const int seg = tid / kFIn, r = tid - seg * kFIn;
            const float2 ref = S.ref[seg * kRow / kFH][c];
            float2 s01[kRow], s23[kRow];
            float s4[kRow];
#pragma unroll
            for (int j = 0; j < kRow; ++j) {
                s01[j] = s23[j] = make_float2(0.f, 0.f);
                s4[j] = 0.f;
            }
#pragma unroll
            for (int t = 0; t < kRow + 2 * kR; ++t) {
                const float2 in = S.in[c][r][seg * kRow + t];
                const float2 v = make_float2(in.x - ref.x, in.y - ref.y);
                const float2 vv = mul2(v, v);
                const float xy = v.x * v.y;
#pragma unroll
                for (int j = 0; j < kRow; ++j)
                    if (t - j >= 0 && t - j <= 2 * kR) {
                        const float w = win.w[t - j];
                        s01[j] = fma2(make_float2(w, w), v, s01[j]);
                        s23[j] = fma2(make_float2(w, w), vv, s23[j]);
                        s4[j] = fmaf(w, xy, s4[j]);
                    }
            }
#pragma unroll
            for (int j = 0; j < kRow; ++j) {
                S.h01[r][seg * kRow + j] = s01[j];
                S.h23[r][seg * kRow + j] = s23[j];
                S.h4[r][seg * kRow + j] = s4[j];
            }
        }
        __syncthreads();
        float2 m01[kCol], m23[kCol];
        float m4[kCol];
#pragma unroll
        for (int j = 0; j < kCol; ++j) {
            m01[j] = m23[j] = make_float2(0.f, 0.f);
            m4[j] = 0.f;
        }
#pragma unroll
        for (int t = 0; t < kCol + 2 * kR; ++t) {
            const float2 a = S.h01[ty + t][tx], b = S.h23[ty + t][tx];
            const float d = S.h4[ty + t][tx];
#pragma unroll
            for (int j = 0; j < kCol; ++j)
                if (t - j >= 0 && t - j <= 2 * kR) {
                    const float w = win.w[t - j];
                    m01[j] = fma2(make_float2(w, w), a, m01[j]);
                    m23[j] = fma2(make_float2(w, w), b, m23[j]);
                    m4[j] = fmaf(w, d, m4[j]);
                }
        }
        const float rx = S.ref[tx / kFH][c].x, ry = S.ref[tx / kFH][c].y;
#pragma unroll
        for (int j = 0; j < kCol; ++j) {
            const int py = y0 + ty + j;
            if (px >= W || py >= H) continue;
            const float sxx = m23[j].x - m01[j].x * m01[j].x, syy = m23[j].y - m01[j].y * m01[j].y;
            const float sxy = m4[j] - m01[j].x * m01[j].y;
            const float mx = m01[j].x + rx, my = m01[j].y + ry;
            const float A = 2.0f * mx * my + kC1, B = 2.0f * sxy + kC2;
            const float Cc = mx * mx + my * my + kC1, D = sxx + syy + kC2;
            const float iCD = 1.0f / (Cc * D);
            const float Sv = A * B * iCD;
            const float g2 = -Sv / D;
            const float g3 = 2.0f * A * iCD;
            const float g1 = 2.0f * my * B * iCD - 2.0f * mx * Sv / Cc - 2.0f * mx * g2 - my * g3;
            const size_t o = (size_t)py * W + px;
            G[(3 * c + 0) * plane + o] = g1;
            G[(3 * c + 1) * plane + o] = g2;
            G[(3 * c + 2) * plane + o] = g3;
            acc += (1.0f - lam) * (1.0f - Sv);
        }
        __syncthreads();   // the next channel's row pass overwrites the row sums
    }
    const float t = block_sum<kFThreads>(acc, S.red);
    if (tid == 0) {
        atomicAdd(&total->sum, (double)t * (double)inv_n);
        __threadfence();
        if (atomicAdd(&total->done, 1u) == gridDim.x * gridDim.y - 1) {
            __threadfence();
            *loss = (float)atomicAdd(&total->sum, 0.0);
        }
    }
}

struct BwdMem {
    float2 in01[kIn][kIn + 1];       // planes G1, G2 of a channel,
    float in2[kIn][kIn + 1];         // G3
    float2 h01[kIn][kT + 1];         // and their row sums
    float h2[kIn][kT + 1];
};

__global__ void __launch_bounds__(kThreads) ssim_bwd_kernel(const float4 *__restrict__ img, const float4 *__restrict__ tgt,
                                                            int H, int W, float lam, float inv_n, Window win,
                                                            const float *__restrict__ G, float4 *__restrict__ dL) {
    __shared__ BwdMem S;
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * kT, y0 = blockIdx.y * kT;
    const size_t plane = (size_t)H * W;
    const int tx = tid & 31, ty = (tid >> 5) * kCol;
    const int px = x0 + tx;
    float out[3][kCol];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        for (int i = tid; i < kIn * kIn; i += kThreads) {
            const int ly = i / kIn, lx = i - ly * kIn;
            const int gx = x0 - kR + lx, gy = y0 - kR + ly;
            const bool in = gx >= 0 && gx < W && gy >= 0 && gy < H;
            const size_t o = (size_t)gy * W + gx;
            S.in01[ly][lx] = in ? make_float2(G[(3 * c + 0) * plane + o], G[(3 * c + 1) * plane + o]) : make_float2(0.f, 0.f);
            S.in2[ly][lx] = in ? G[(3 * c + 2) * plane + o] : 0.0f;
        }
        __syncthreads();
        if (tid < kRowTasks) {
            const int seg = tid / kIn, r = tid - seg * kIn;
            float2 s01[kRow];
            float s2[kRow];
#pragma unroll
            for (int j = 0; j < kRow; ++j) {
                s01[j] = make_float2(0.f, 0.f);
                s2[j] = 0.f;
            }
#pragma unroll
            for (int t = 0; t < kRow + 2 * kR; ++t) {
                const float2 v = S.in01[r][seg * kRow + t];
                const float u = S.in2[r][seg * kRow + t];
#pragma unroll
                for (int j = 0; j < kRow; ++j)
                    if (t - j >= 0 && t - j <= 2 * kR) {
                        const float w = win.w[t - j];
                        s01[j] = fma2(make_float2(w, w), v, s01[j]);
                        s2[j] = fmaf(w, u, s2[j]);
                    }
            }
#pragma unroll
            for (int j = 0; j < kRow; ++j) {
                S.h01[r][seg * kRow + j] = s01[j];
                S.h2[r][seg * kRow + j] = s2[j];
            }
        }
        __syncthreads();
        float2 b01[kCol];
        float b2[kCol];
#pragma unroll
        for (int j = 0; j < kCol; ++j) {
            b01[j] = make_float2(0.f, 0.f);
            b2[j] = 0.f;
        }
#pragma unroll
        for (int t = 0; t < kCol + 2 * kR; ++t) {
            const float2 a = S.h01[ty + t][tx];
            const float d = S.h2[ty + t][tx];
#pragma unroll
            for (int j = 0; j < kCol; ++j)
                if (t - j >= 0 && t - j <= 2 * kR) {
                    const float w = win.w[t - j];
                    b01[j] = fma2(make_float2(w, w), a, b01[j]);
                    b2[j] = fmaf(w, d, b2[j]);
                }
        }
#pragma unroll
        for (int j = 0; j < kCol; ++j) {
            const int py = y0 + ty + j;
            out[c][j] = 0.0f;
            if (px >= W || py >= H) continue;
            const size_t o = 4 * ((size_t)py * W + px) + c;
            const float x = __ldg(reinterpret_cast<const float *>(img) + o), y = __ldg(reinterpret_cast<const float *>(tgt) + o);
            const float dS = (b01[j].x + 2.0f * x * b01[j].y + y * b2[j]) * inv_n;
            const float d = x - y;
            const float sg1 = d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f);
            out[c][j] = lam * sg1 * inv_n - (1.0f - lam) * dS;
        }
        // (the next channel's staging writes other words than the column pass reads; its row pass comes
        // after a barrier)
    }
#pragma unroll
    for (int j = 0; j < kCol; ++j) {
        const int py = y0 + ty + j;
        if (px < W && py < H) dL[(size_t)py * W + px] = make_float4(out[0][j], out[1][j], out[2][j], 0.0f);
    }
}

Window make_window() {
    Window w;
    double g[2 * kR + 1], z = 0.0;
    for (int t = -kR; t <= kR; ++t) {
        g[t + kR] = std::exp(-(double)(t * t) / (2.0 * 1.5 * 1.5));
        z += g[t + kR];
    }
    for (int t = 0; t <= 2 * kR; ++t) w.w[t] = (float)(g[t] / z);
    return w;
}

}  // namespace

size_t ssim_scratch_bytes(int H, int W) { return (size_t)9 * sizeof(float) * (size_t)H * (size_t)W; }   // the planes

cudaError_t launch_ssim_loss(const float *img, const float *tgt, int H, int W, float lam, float *dL, float *loss,
                             char *scratch, cudaStream_t st) {
    if (H == 0 || W == 0) return cudaMemsetAsync(loss, 0, sizeof(float), st);
    LossSum *total = reinterpret_cast<LossSum *>(scratch);
    float *G = reinterpret_cast<float *>(total + 1);
    cudaError_t e = cudaMemsetAsync(total, 0, sizeof(LossSum), st);
    if (e != cudaSuccess) return e;
    const dim3 grid((W + kT - 1) / kT, (H + kT - 1) / kT), fwd_grid(grid.x, (H + kFH - 1) / kFH);
    const float inv_n = (float)(1.0 / (3.0 * (double)H * (double)W));
    const Window win = make_window();
    ssim_fwd_kernel<<<fwd_grid, kFThreads, 0, st>>>(reinterpret_cast<const float4 *>(img), reinterpret_cast<const float4 *>(tgt),
                                            H, W, lam, inv_n, win, G, total, loss);
    ssim_bwd_kernel<<<grid, kThreads, 0, st>>>(reinterpret_cast<const float4 *>(img), reinterpret_cast<const float4 *>(tgt),
                                            H, W, lam, inv_n, win, G, reinterpret_cast<float4 *>(dL));
    return cudaGetLastError();
}

}  // namespace ms
