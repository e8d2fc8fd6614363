// Image loss of the training objective (Sec. 4.4, total loss): the L1 term and
// the SSIM term (structural similarity, Wang et al. 2004: local means,
// variances and covariance under an 11x11 Gaussian window of standard
// deviation 1.5, constants C1 = 0.01^2, C2 = 0.03^2), with their gradient
// with respect to the rendered image.  The window extends past the image
// border with zeros, so every map has the image's size.
//
//   k_ssim_forward   per 32x54 tile of one channel: stage x, y and a 5-pixel
//                    halo in shared memory, blur x, y, x^2, y^2, xy along rows
//                    and then columns, form the SSIM map S and the partial
//                    derivatives of w_ssim * (1 - mean S) with respect to the
//                    three local moments mu_x, E[x^2], E[xy]; sum S and |x - y|.
//   k_ssim_backward  blurs the three derivative maps (the window is symmetric,
//                    so the adjoint of the zero-padded blur is the same blur)
//                    and combines them with x and y; adds the L1 gradient.
//
// Both are bound by the FP32 pipe: 110 (66) FMA per pixel for the blurs, 1.19
// times the row half for the vertical halo.  A thread blurs four pixels of a row
// (14 inputs, 16-byte shared loads) and then seven of a column (17 inputs), so
// an input is loaded once per 3 to 4 taps rather than per tap, and x with y
// (x^2 with y^2, and the derivative maps in a pair) go through one paired FMA,
// which rounds each half as fmaf does.  64 staged rows are two rounds of 256
// threads without a remainder; the row strides put the eight rows of a load or
// store phase into distinct banks.  Sums over pixels run in float pairs (two-sum)
// and only the tiles' totals in FP64, of which this chip has 1/64 of the FP32
// rate: summed pixel by pixel in FP64, a pass without the gradient takes 76 us instead
// of 57, and both give the exact mean of |x - y| (images in [0, 1], 64x48 to 1920x1080).  1920x1080x3, forward / backward: 118 / 85 us with one output per thread
// and step and FP64 sums, 75 / 42 us now (3 CTAs per SM; 66 forward with one shared
// reciprocal instead of seven quotients a pixel).
#include "adr_internal.cuh"

namespace adr {
namespace {

constexpr int kLW = 32;                  // output tile
constexpr int kLTall = 54;
constexpr int kLR = 5;                   // window radius (11 taps)
constexpr int kTaps = 2 * kLR + 1;
constexpr int kLRows = kLTall + 2 * kLR; // staged rows: 64, 8 per warp
constexpr int kLCols = kLW + 2 * kLR;
constexpr int kLThreads = 256;
constexpr int kLStage = (kLRows * kLCols + kLThreads - 1) / kLThreads;   // staged pixels per thread
constexpr int kQuad = 4;                 // pixels of a row per thread and round
constexpr int kRun = 7;                  // pixels of a column per thread
constexpr int kPairStride = 46;          // float2 per staged row: 368 B, 8 rows on distinct 16-byte banks
constexpr int kFloatStride = 44;         // floats per staged row: 176 B, likewise
constexpr int kPairOut = kLW + 2;        // float2 per row-blurred row: 272 B
constexpr int kFloatOut = kLW + 4;       // floats per row-blurred row: 144 B
static_assert(kLRows == 8 * (kLThreads / 32) && kLW == 2 * kQuad * 4, "two rounds of 8 rows x 4 quads a warp");
static_assert(kRun * (kLThreads / 32) >= kLTall, "a warp per run of rows");
constexpr float kC1 = 0.01f * 0.01f;
constexpr float kC2 = 0.03f * 0.03f;

struct alignas(16) ForwardShared {
    float2 xy[kLRows * kPairStride];
    float2 m[kLRows * kPairOut];         // row-blurred (x, y)
    float2 mm[kLRows * kPairOut];        // row-blurred (x^2, y^2)
    float p[kLRows * kFloatOut];         // row-blurred xy
    float2 red[2][kLThreads / 32];       // L1 and SSIM sums
};
struct alignas(16) BackwardShared {
    float2 ab[kLRows * kPairStride];     // derivative maps (mu, xx)
    float c[kLRows * kFloatStride];      // xy
    float2 hab[kLRows * kPairOut];
    float hc[kLRows * kFloatOut];
};

// (hi, lo) += v with hi + lo kept to about twice FP32's precision.
__device__ __forceinline__ void pair_add(float2& acc, float v) {
    const float s = __fadd_rn(acc.x, v), b = __fsub_rn(s, acc.x);
    acc.y = __fadd_rn(acc.y, __fadd_rn(__fsub_rn(acc.x, __fsub_rn(s, b)), __fsub_rn(v, b)));
    acc.x = s;
}
__device__ __forceinline__ float2 pair_sum(float2 a, float2 b) {
    pair_add(a, b.x);
    a.y = __fadd_rn(a.y, b.y);
    return a;
}

__global__ void __launch_bounds__(kLThreads, 3)
k_ssim_forward(const float* __restrict__ img, const float* __restrict__ ref, int H, int W,
               LossWindow win, float g_scale, float* __restrict__ g_mu,
               float* __restrict__ g_xx, float* __restrict__ g_xy, double* __restrict__ stats) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ForwardShared& sm = *reinterpret_cast<ForwardShared*>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int X0 = blockIdx.x * kLW, Y0 = blockIdx.y * kLTall;
    const uint32_t channel = blockIdx.z * (uint32_t)(H * W);   // at most 2^31 elements in all
    const float* xs = img + channel;
    const float* ys = ref + channel;
    // All of a thread's loads are issued before the first is stored: their
    // latency shows once per tile.
    float2 v[kLStage];
#pragma unroll
    for (int u = 0; u < kLStage; ++u) {
        const int i = u * kLThreads + threadIdx.x, r = i / kLCols, q = i % kLCols;
        const int gy = Y0 - kLR + r, gx = X0 - kLR + q;
        const uint32_t o = (uint32_t)(gy * W + gx);
        v[u] = make_float2(0.f, 0.f);
        if (gy >= 0 && gy < H && gx >= 0 && gx < W && i < kLRows * kLCols) v[u] = make_float2(xs[o], ys[o]);
    }
#pragma unroll
    for (int u = 0; u < kLStage; ++u) {
        const int i = u * kLThreads + threadIdx.x;
        if (i < kLRows * kLCols) sm.xy[(i / kLCols) * kPairStride + i % kLCols] = v[u];
    }
    __syncthreads();
    // Rows: warp w blurs rows 8 w .. 8 w + 7, lane l row l mod 8, quad l / 8 (+ 4).
#pragma unroll 1
    for (int round = 0; round < 2; ++round) {
        const int r = 8 * warp + (lane & 7), q0 = kQuad * (4 * round + (lane >> 3));
        const float4* in = reinterpret_cast<const float4*>(sm.xy + r * kPairStride + q0);
        float2 m[kQuad], mm[kQuad];
        float p[kQuad];
#pragma unroll
        for (int o = 0; o < kQuad; ++o) {
            m[o] = mm[o] = make_float2(0.f, 0.f);
            p[o] = 0.f;
        }
#pragma unroll
        for (int j2 = 0; j2 < (kQuad + kTaps - 1) / 2; ++j2) {
            const float4 v = in[j2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = 2 * j2 + h;
                const float2 xy = h ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
                const float2 sq = fmul2(xy, xy);
                const float pr = __fmul_rn(xy.x, xy.y);
#pragma unroll
                for (int o = 0; o < kQuad; ++o) {
                    const int k = j - o;
                    if (k < 0 || k >= kTaps) continue;
                    const float2 w = make_float2(win.w[k], win.w[k]);
                    m[o] = ffma2(w, xy, m[o]);
                    mm[o] = ffma2(w, sq, mm[o]);
                    p[o] = fmaf(w.x, pr, p[o]);
                }
            }
        }
        float4* om = reinterpret_cast<float4*>(sm.m + r * kPairOut + q0);
        float4* omm = reinterpret_cast<float4*>(sm.mm + r * kPairOut + q0);
#pragma unroll
        for (int o = 0; o < kQuad; o += 2) {
            om[o / 2] = make_float4(m[o].x, m[o].y, m[o + 1].x, m[o + 1].y);
            omm[o / 2] = make_float4(mm[o].x, mm[o].y, mm[o + 1].x, mm[o + 1].y);
        }
        *reinterpret_cast<float4*>(sm.p + r * kFloatOut + q0) = make_float4(p[0], p[1], p[2], p[3]);
    }
    __syncthreads();
    // Columns: warp w outputs rows 7 w .. 7 w + 6, lane l column l.
    float2 m[kRun], mm[kRun];
    float p[kRun];
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
        m[o] = mm[o] = make_float2(0.f, 0.f);
        p[o] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < kRun + kTaps - 1; ++j) {
        const int r = min(kRun * warp + j, kLRows - 1);   // past the last output row only
        const float2 a = sm.m[r * kPairOut + lane], aa = sm.mm[r * kPairOut + lane];
        const float ab = sm.p[r * kFloatOut + lane];
#pragma unroll
        for (int o = 0; o < kRun; ++o) {
            const int k = j - o;
            if (k < 0 || k >= kTaps) continue;
            const float2 w = make_float2(win.w[k], win.w[k]);
            m[o] = ffma2(w, a, m[o]);
            mm[o] = ffma2(w, aa, mm[o]);
            p[o] = fmaf(w.x, ab, p[o]);
        }
    }
    float2 ssim_sum = make_float2(0.f, 0.f), l1_sum = make_float2(0.f, 0.f);
    const int gx = X0 + lane;
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
        const int r = kRun * warp + o, gy = Y0 + r;
        if (r >= kLTall || gy >= H || gx >= W) continue;
        const float mx = m[o].x, my = m[o].y;
        const float vx = mm[o].x - mx * mx, vy = mm[o].y - my * my, cxy = p[o] - mx * my;
        const float A1 = 2.f * mx * my + kC1, A2 = 2.f * cxy + kC2;
        const float B1 = mx * mx + my * my + kC1, B2 = vx + vy + kC2;
        const float S = (A1 * A2) / (B1 * B2);
        const float2 xy = sm.xy[(r + kLR) * kPairStride + lane + kLR];
        pair_add(ssim_sum, S);
        pair_add(l1_sum, fabsf(xy.x - xy.y));
        if (g_mu) {
            // dS/dmu_x, dS/dE[x^2], dS/dE[xy] at this pixel, times d loss / dS.
            // A quotient each: their sums cancel in the gradient, and one shared
            // reciprocal put it up to 1e-6 further from FP64.
            const float d_mu = S * (2.f * my / A1 - 2.f * my / A2 - 2.f * mx / B1 + 2.f * mx / B2);
            const float d_xx = -S / B2;
            const float d_xy = 2.f * S / A2;
            const uint32_t at = channel + (uint32_t)(gy * W + gx);
            g_mu[at] = g_scale * d_mu;
            g_xx[at] = g_scale * d_xx;
            g_xy[at] = g_scale * d_xy;
        }
    }
    // The tile's sums, still as float pairs; FP64 for the global ones only.
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ssim_sum = pair_sum(ssim_sum, make_float2(__shfl_xor_sync(0xffffffffu, ssim_sum.x, o),
                                                  __shfl_xor_sync(0xffffffffu, ssim_sum.y, o)));
        l1_sum = pair_sum(l1_sum, make_float2(__shfl_xor_sync(0xffffffffu, l1_sum.x, o),
                                              __shfl_xor_sync(0xffffffffu, l1_sum.y, o)));
    }
    if (lane == 0) sm.red[0][warp] = l1_sum;
    if (lane == 0) sm.red[1][warp] = ssim_sum;
    // An infinite difference, or a sum over FP32's range, makes the pairs' second words NaN:
    // such a tile's |x - y| are summed again, in FP64.
    const bool beyond = __syncthreads_or(!(l1_sum.x < 4e37f));   // eight warps' sums stay finite
    if (threadIdx.x < 2) {
        float2 t = make_float2(0.f, 0.f);
        for (int w = 0; w < kLThreads / 32; ++w) t = pair_sum(t, sm.red[threadIdx.x][w]);
        if (!beyond || threadIdx.x == 1) atomicAdd(stats + threadIdx.x, isfinite(t.x) ? (double)t.x + (double)t.y : (double)t.x);
    }
    if (!beyond) return;
    double sum = 0.0;
    for (int i = threadIdx.x; i < kLW * kLTall; i += kLThreads) {
        const int r = i / kLW, q = i % kLW;
        if (Y0 + r >= H || X0 + q >= W) continue;
        const float2 xy = sm.xy[(r + kLR) * kPairStride + q + kLR];
        sum += (double)fabsf(xy.x - xy.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) atomicAdd(stats, sum);
}

__global__ void __launch_bounds__(kLThreads, 3)
k_ssim_backward(const float* __restrict__ img, const float* __restrict__ ref, int H, int W,
                LossWindow win, const float* __restrict__ g_mu, const float* __restrict__ g_xx,
                const float* __restrict__ g_xy, float l1_scale, float* __restrict__ dl_dimg) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BackwardShared& sm = *reinterpret_cast<BackwardShared*>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int X0 = blockIdx.x * kLW, Y0 = blockIdx.y * kLTall;
    const uint32_t channel = blockIdx.z * (uint32_t)(H * W);   // at most 2^31 elements in all
    {
        float2 v[kLStage];
        float w[kLStage];
#pragma unroll
        for (int u = 0; u < kLStage; ++u) {
            const int i = u * kLThreads + threadIdx.x, r = i / kLCols, q = i % kLCols;
            const int gy = Y0 - kLR + r, gx = X0 - kLR + q;
            const uint32_t o = channel + (uint32_t)(gy * W + gx);
            v[u] = make_float2(0.f, 0.f);
            w[u] = 0.f;
            if (gy >= 0 && gy < H && gx >= 0 && gx < W && i < kLRows * kLCols) {
                v[u] = make_float2(g_mu[o], g_xx[o]);
                w[u] = g_xy[o];
            }
        }
#pragma unroll
        for (int u = 0; u < kLStage; ++u) {
            const int i = u * kLThreads + threadIdx.x;
            if (i < kLRows * kLCols) {
                sm.ab[(i / kLCols) * kPairStride + i % kLCols] = v[u];
                sm.c[(i / kLCols) * kFloatStride + i % kLCols] = w[u];
            }
        }
    }
    __syncthreads();
    // this thread's output pixels, while the blurs run
    const int gx = X0 + lane;
    float px[kRun], py[kRun];
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
        const int r = kRun * warp + o, gy = Y0 + r;
        const uint32_t at = channel + (uint32_t)(gy * W + gx);
        px[o] = py[o] = 0.f;
        if (r < kLTall && gy < H && gx < W) {
            px[o] = img[at];
            py[o] = ref[at];
        }
    }
#pragma unroll 1
    for (int round = 0; round < 2; ++round) {   // rows, as in k_ssim_forward
        const int r = 8 * warp + (lane & 7), q0 = kQuad * (4 * round + (lane >> 3));
        const float4* in_ab = reinterpret_cast<const float4*>(sm.ab + r * kPairStride + q0);
        const float4* in_c = reinterpret_cast<const float4*>(sm.c + r * kFloatStride + q0);
        float2 ab[kQuad];
        float c[kQuad];
#pragma unroll
        for (int o = 0; o < kQuad; ++o) {
            ab[o] = make_float2(0.f, 0.f);
            c[o] = 0.f;
        }
#pragma unroll
        for (int j4 = 0; j4 < (kQuad + kTaps - 1 + 3) / 4; ++j4) {
            const float4 vc = in_c[j4];   // up to 2 past the 14 inputs, inside the row's stride
            const float cs[4] = {vc.x, vc.y, vc.z, vc.w};
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                const int j2 = 2 * j4 + h2;
                if (2 * j2 >= kQuad + kTaps - 1) continue;
                const float4 v = in_ab[j2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = 2 * j2 + h;
                    const float2 t = h ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
#pragma unroll
                    for (int o = 0; o < kQuad; ++o) {
                        const int k = j - o;
                        if (k < 0 || k >= kTaps) continue;
                        ab[o] = ffma2(make_float2(win.w[k], win.w[k]), t, ab[o]);
                        c[o] = fmaf(win.w[k], cs[2 * h2 + h], c[o]);
                    }
                }
            }
        }
        float4* oab = reinterpret_cast<float4*>(sm.hab + r * kPairOut + q0);
        oab[0] = make_float4(ab[0].x, ab[0].y, ab[1].x, ab[1].y);
        oab[1] = make_float4(ab[2].x, ab[2].y, ab[3].x, ab[3].y);
        *reinterpret_cast<float4*>(sm.hc + r * kFloatOut + q0) = make_float4(c[0], c[1], c[2], c[3]);
    }
    __syncthreads();
    float2 ab[kRun];
    float c[kRun];
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
        ab[o] = make_float2(0.f, 0.f);
        c[o] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < kRun + kTaps - 1; ++j) {
        const int r = min(kRun * warp + j, kLRows - 1);
        const float2 t = sm.hab[r * kPairOut + lane];
        const float u = sm.hc[r * kFloatOut + lane];
#pragma unroll
        for (int o = 0; o < kRun; ++o) {
            const int k = j - o;
            if (k < 0 || k >= kTaps) continue;
            ab[o] = ffma2(make_float2(win.w[k], win.w[k]), t, ab[o]);
            c[o] = fmaf(win.w[k], u, c[o]);
        }
    }
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
        const int r = kRun * warp + o, gy = Y0 + r;
        if (r >= kLTall || gy >= H || gx >= W) continue;
        const uint32_t at = channel + (uint32_t)(gy * W + gx);
        const float x = px[o], y = py[o];
        const float d = x - y;
        const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
        dl_dimg[at] = ab[o].x + 2.f * x * ab[o].y + y * c[o] + l1_scale * sgn;
    }
}

// The means and, where asked for, the loss: formed here, as one more launch over
// one value costs a caller as much as a pass over a small image.
__global__ void k_loss_finalize(double* stats, double count, double w_l1, double w_ssim, float* loss) {
    const double l1 = stats[0] / count, ssim = stats[1] / count;
    stats[0] = l1;
    stats[1] = ssim;
    if (loss) *loss = (float)__dadd_rn(__dmul_rn(w_l1, l1), __dmul_rn(w_ssim, 1.0 - ssim));
}

}  // namespace

void launch_image_loss(const float* img, const float* ref, int channels, int H, int W,
                       const LossWindow& win, double w_l1, double w_ssim, double* stats, float* loss,
                       float* dl_dimg, float* scratch, cudaStream_t stream) {
    const dim3 grid((W + kLW - 1) / kLW, (H + kLTall - 1) / kLTall, channels);
    const double count = (double)channels * H * W;
    const size_t n = (size_t)channels * H * W;
    float* g_mu = dl_dimg ? scratch : nullptr;
    float* g_xx = dl_dimg ? scratch + n : nullptr;
    float* g_xy = dl_dimg ? scratch + 2 * n : nullptr;
    // more than 48 KB of shared memory has to be asked for, per device
    cudaFuncSetAttribute(k_ssim_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ForwardShared));
    cudaFuncSetAttribute(k_ssim_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BackwardShared));
    cudaMemsetAsync(stats, 0, 2 * sizeof(double), stream);
    // loss = w_l1 * mean|x - y| + w_ssim * (1 - mean S): d loss / dS = -w_ssim / count
    k_ssim_forward<<<grid, kLThreads, sizeof(ForwardShared), stream>>>(img, ref, H, W, win, (float)(-(float)w_ssim / count),
                                                   g_mu, g_xx, g_xy, stats);
    if (dl_dimg)
        k_ssim_backward<<<grid, kLThreads, sizeof(BackwardShared), stream>>>(img, ref, H, W, win, g_mu, g_xx, g_xy,
                                                        (float)((float)w_l1 / count), dl_dimg);
    k_loss_finalize<<<1, 1, 0, stream>>>(stats, count, w_l1, w_ssim, loss);
}

}  // namespace adr
