// Adaptive spatial smoothing (Sec. 3.4, Eqs. eq:lem_fmlp and eq:lem_loss_mlp;
// supplementary Tab. pemlp): per Gaussian s_MLP = MLP(p) (positional encoding
// of frequency 0 = the position), MLP 3 -> 128 -> 128 -> 128 -> 8 (ReLU x 3),
//   L_smo = |s_MLP - s_G*| + max(u*, w_s) |s_MLP* - s_G|   (* = stop gradient),
// its mean over the Gaussians times lambda_smo, the gradient of every MLP
// parameter (through the first term) and of s_G (through the second).
//
// smooth_kernel: persistent, one CTA per SM, tiles of 128 Gaussians one after
// another.  Four warpgroups serve the tile's 128 rows (TMEM lanes), each
// taking 32 of every 128-column epilogue's columns; the loss epilogue is
// warpgroup 0's.  A warp of its own issues each tcgen05.mma round (an epilogue
// warp that does is held up while the MMAs queue); after it completes, the
// warpgroups run its epilogue (bias and ReLU, or the ReLU's mask, BF16 into
// shared memory):
//   forward  H1 = relu(X W1^T + b1), H2, H3, Z = H3 W4^T + b4 (FP32 accumulation)
//   loss     per row: diff = Z - s_G, n = |diff|; dZ = lambda/n_total diff/n;
//            d_feat -= lambda/n_total max(u, w_s) diff/n (added to the caller's array)
//   backward dH3 = (dZ W4) o [H3 > 0], dH2 = (dH3 W3) o [H2 > 0], dH1 = ...,
//            in a buffer of their own and in H3's, so that a round's weight
//            gradients, which read the layer outputs, run under the epilogue of
//            its input gradient (1M Gaussians 0.490 -> 0.467 ms; with
//            the MMA warp 0.427).  Weight gradients
//            dW = dH^T H_prev accumulate in
//            TMEM over all of a CTA's tiles (MMAs reading both operands
//            MN-major from the row-major activation buffers, no transposed
//            copies); the bias sums come from MMAs against a ones column (b2, b3),
//            the ones column of X (b1) and a warp transposition (b4).
// At the end each CTA adds its accumulators to the caller's gradients with
// atomics.  Every wait is bounded; on a timeout the kernel records it,
// stops issuing work, waits (bounded) for its MMAs and frees its TMEM.
#include "tc_common.cuh"

namespace leg {

__device__ int g_smooth_error;

namespace {
using namespace tc;

constexpr int kH = 128, kS = 8;
constexpr int kParts = 4;                    // warpgroups per CTA
constexpr int kEpiWarps = 4 * kParts;
constexpr int kThreadsS = 32 * (kEpiWarps + 1);   // and the MMA warp
// TMEM columns
constexpr uint32_t kAcc = 0, kDW2 = 128, kDW3 = 256, kDW1 = 384, kDW4 = 400, kDB2 = 416, kDB3 = 432;

struct SmoothArgs {
    int n, ntiles;
    const float *means, *feat, *unc;
    const float *W1, *b1, *W2, *b2, *W3, *b3, *W4, *b4;
    float w_s, scale;              // scale = lambda_smo / n
    float* loss;
    float* d_feat;
    int d_feat_stride;
    float* s_mlp;                  // nullable
    float *dW1, *db1, *dW2, *db2, *dW3, *db3, *dW4, *db4;
};

// Shared-memory plan (canonical no-swizzle BF16 buffers; byte offsets).
constexpr uint32_t kOW1 = 0;                                 // [128][16]
constexpr uint32_t kOW2 = kOW1 + sbuf_bytes(128, 16);        // [128][128]
constexpr uint32_t kOW3 = kOW2 + sbuf_bytes(128, 128);
constexpr uint32_t kOW4 = kOW3 + sbuf_bytes(128, 128);       // [16][128]
constexpr uint32_t kOX = kOW4 + sbuf_bytes(16, 128);         // [2][128][16], column 3 = 1 (tiles alternate)
constexpr uint32_t kOH1 = kOX + 2 * sbuf_bytes(128, 16);     // [128][128]
constexpr uint32_t kOH2 = kOH1 + sbuf_bytes(128, 128);
constexpr uint32_t kOH3 = kOH2 + sbuf_bytes(128, 128);       // H3, later dH2
constexpr uint32_t kOD = kOH3 + sbuf_bytes(128, 128);        // dH3, later dH1
constexpr uint32_t kODZ = kOD + sbuf_bytes(128, 128);        // [128][16]
constexpr uint32_t kOE = kODZ + sbuf_bytes(128, 16);         // [128][16], column 0 = 1
constexpr uint32_t kOB = kOE + sbuf_bytes(128, 16);          // biases FP32: b1, b2, b3 (128 each), b4 (8)
constexpr uint32_t kOBar = kOB + (3 * kH + 16) * 4;
constexpr uint32_t kSmoothSmem = kOBar + 48 + 1024;
static_assert(kSmoothSmem <= 227 * 1024, "smoothing shared memory");

struct Ctx {
    unsigned char* sm;
    uint32_t s0;                   // shared address of sm
    // a round's operands written, one arrival per epilogue warp (even and odd rounds, so that a warp that runs
    // ahead from the last round of a tile into the next tile's first one does not count for another); its result
    uint64_t *ready, *done;
    uint32_t* tslot;
    uint32_t phase;
    uint32_t tmem, lanef;
    int row;
    int part;                      // warpgroup: columns [32 part, 32 part + 32) of each hidden epilogue
};

// This warp's shared-memory writes are visible to the tensor core and its TMEM
// reads ordered before the next MMAs; then wait for those.
__device__ __forceinline__ bool next_round(Ctx& c, int round)
{
    fence_proxy_async();
    fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(c.ready + (round & 1));
    const bool ok = warp_agree(mbar_wait(c.done, c.phase));
    c.phase ^= 1u;
    fence_after();
    return ok;
}

// This warpgroup's 32 columns of the epilogue of a 128-column hidden layer:
// relu(acc + b) in BF16 into H.
__device__ __forceinline__ void hidden_epilogue(const Ctx& c, const float* b, uint32_t hoff)
{
    float v[16];
    uint32_t w[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int col = 32 * c.part + 16 * q;
        tmem_ld16(c.tmem + c.lanef + kAcc + col, v);
        relu16(v, b + col, w);
        sts_row16(c.s0 + hoff + sbuf_off(c.row, col, kH), w);
    }
}

// This warpgroup's 32 columns of a backward epilogue: dH = acc o [H > 0], BF16 into dst.
__device__ __forceinline__ void grad_epilogue(const Ctx& c, uint32_t hoff, uint32_t dst)
{
    float v[16];
    uint32_t w[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int col = 32 * c.part + 16 * q;
        const uint32_t at = c.s0 + sbuf_off(c.row, col, kH);
        tmem_ld16(c.tmem + c.lanef + kAcc + col, v);
        relu_mask16(v, at + hoff, w);
        sts_row16(at + dst, w);
    }
}

// K-major descriptor of a C-column buffer at shared offset off (rows from 0).
__device__ __forceinline__ uint64_t kd(uint32_t s0, uint32_t off, int C) { return kdesc_at(s0 + off, C, 0, 0); }
// MN-major descriptor (rows = K) of a C-column buffer.
__device__ __forceinline__ uint64_t md(uint32_t s0, uint32_t off, int C) { return mndesc_at(s0 + off, C, 0, 0); }

// One MMA round, issued by the MMA warp's elected lane.  K steps of 16 move the
// start address by 16 units (K-major) or 2C units (MN-major over a C-column
// buffer).  The commit follows the MMAs whose result the next epilogue reads;
// the weight gradients behind it run under that epilogue (they are complete by
// the next round's commit, which is before anything they read is written again)
// and the last round, dW1, under the next tile's first one.  x: this tile's X.
__device__ __forceinline__ void issue(const Ctx& c, int round, bool first_tile, uint32_t x)
{
    if (!elect_one()) return;
    const uint32_t s0 = c.s0, t = c.tmem;
    const uint32_t keep = first_tile ? 0u : 1u;
    switch (round) {
        case 0:   // H1 pre-activation = X W1^T
            mma(t + kAcc, kd(s0, x, 16), kd(s0, kOW1, 16), idesc_bf16(kH, false, false), 0u);
            commit(c.done);
            break;
        case 1:   // H2 = H1 W2^T
        case 2: { // H3 = H2 W3^T
            const uint64_t a = kd(s0, round == 1 ? kOH1 : kOH2, kH), b = kd(s0, round == 1 ? kOW2 : kOW3, kH);
#pragma unroll
            for (int k = 0; k < 8; ++k) mma(t + kAcc, a + 16 * k, b + 16 * k, idesc_bf16(kH, false, false), k > 0);
            commit(c.done);
            break;
        }
        case 3: { // Z = H3 W4^T (N = 16, 8 used)
            const uint64_t a = kd(s0, kOH3, kH), b = kd(s0, kOW4, kH);
#pragma unroll
            for (int k = 0; k < 8; ++k) mma(t + kAcc, a + 16 * k, b + 16 * k, idesc_bf16(16, false, false), k > 0);
            commit(c.done);
            break;
        }
        case 4: { // dH3 (pre-mask) = dZ W4; dW4^T += H3^T dZ
            mma(t + kAcc, kd(s0, kODZ, 16), md(s0, kOW4, kH), idesc_bf16(kH, false, true), 0u);
            commit(c.done);
            const uint64_t a = md(s0, kOH3, kH), b = md(s0, kODZ, 16);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(t + kDW4, a + 256 * k, b + 32 * k, idesc_bf16(16, true, true), k > 0 ? 1u : keep);
            break;
        }
        case 5:   // dH2 = dH3 W3; dW3 += dH3^T H2; db3 += dH3^T 1
        case 6: { // dH1 = dH2 W2; dW2 += dH2^T H1; db2 += dH2^T 1
            const uint32_t dh = round == 5 ? kOD : kOH3, w = round == 5 ? kOW3 : kOW2, hp = round == 5 ? kOH2 : kOH1;
            const uint32_t dw = round == 5 ? kDW3 : kDW2, db = round == 5 ? kDB3 : kDB2;
            const uint64_t ak = kd(s0, dh, kH), wm = md(s0, w, kH);
#pragma unroll
            for (int k = 0; k < 8; ++k) mma(t + kAcc, ak + 16 * k, wm + 256 * k, idesc_bf16(kH, false, true), k > 0);
            commit(c.done);
            const uint64_t am = md(s0, dh, kH), hm = md(s0, hp, kH), em = md(s0, kOE, 16);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(t + dw, am + 256 * k, hm + 256 * k, idesc_bf16(kH, true, true), k > 0 ? 1u : keep);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(t + db, am + 256 * k, em + 32 * k, idesc_bf16(16, true, true), k > 0 ? 1u : keep);
            break;
        }
        default: { // dW1 (+ db1 in column 3) += dH1^T X
            const uint64_t am = md(s0, kOD, kH), xm = md(s0, x, 16);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(t + kDW1, am + 256 * k, xm + 32 * k, idesc_bf16(16, true, true), k > 0 ? 1u : keep);
            break;
        }
    }
}

// Sum over the warp's 32 rows of 16 values (recursive halving); lanes 2j, 2j+1 hold column j.
template <int N, int O>
__device__ __forceinline__ void halve16(float* v, bool upper)
{
    constexpr int Hh = N / 2;
#pragma unroll
    for (int i = 0; i < Hh; ++i) {
        const float lo = v[i], hi = v[i + Hh];
        const float recv = __shfl_xor_sync(0xffffffffu, upper ? lo : hi, O);
        v[i] = (upper ? hi : lo) + recv;
    }
}

__device__ __forceinline__ float colsum16(float* v, int lane)
{
    halve16<16, 16>(v, lane & 16);
    halve16<8, 8>(v, lane & 8);
    halve16<4, 4>(v, lane & 4);
    halve16<2, 2>(v, lane & 2);
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

__global__ void __launch_bounds__(kThreadsS, 1) smooth_kernel(SmoothArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    Ctx c;
    c.sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    c.s0 = smem_u32(c.sm);
    c.ready = reinterpret_cast<uint64_t*>(c.sm + kOBar);
    c.done = c.ready + 2;
    uint64_t* const fin = c.ready + 3;
    c.tslot = reinterpret_cast<uint32_t*>(c.sm + kOBar + 32);
    c.phase = 0;
    c.row = threadIdx.x & 127;
    c.part = threadIdx.x >> 7;
    const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    c.lanef = (uint32_t)(32 * (warp & 3)) << 16;
    // weights (BF16, [out][in]), biases (FP32), the ones operand
    sbuf_fill(SBuf{c.sm + kOW1, 16}, 128, a.W1, 3, kH, 3);
    sbuf_fill_rows(SBuf{c.sm + kOW2, kH}, 128, a.W2);
    sbuf_fill_rows(SBuf{c.sm + kOW3, kH}, 128, a.W3);
    sbuf_fill(SBuf{c.sm + kOW4, kH}, 16, a.W4, kH, kS, kH);
    float* bs = reinterpret_cast<float*>(c.sm + kOB);
    for (int i = threadIdx.x; i < 3 * kH + 16; i += blockDim.x)
        bs[i] = i < kH ? a.b1[i] : i < 2 * kH ? a.b2[i - kH] : i < 3 * kH ? a.b3[i - 2 * kH]
              : (i - 3 * kH < kS ? a.b4[i - 3 * kH] : 0.f);
    if (c.part == 0) {
        float v[8] = {1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, z[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        sbuf_store8(SBuf{c.sm + kOE, 16}, c.row, 0, v);
        sbuf_store8(SBuf{c.sm + kOE, 16}, c.row, 8, z);
    }
    if (threadIdx.x == 0) {
        mbar_init(c.ready, kEpiWarps);
        mbar_init(c.ready + 1, kEpiWarps);
        mbar_init(c.done, 1);
        mbar_init(fin, 1);
    }
    if (warp == 0) tmem_alloc(c.tslot, 512);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    c.tmem = warp_uniform(*reinterpret_cast<volatile uint32_t*>(c.tslot));

    const float* b1 = bs;
    const float* b2 = bs + kH;
    const float* b3 = bs + 2 * kH;
    const float* b4 = bs + 3 * kH;
    double lsum = 0.0;                           // one add per row and tile
    float db4acc = 0.f;
    bool ok = true, any = false, odd = false;
    if (warp == kEpiWarps) {
        // every round's operands are ready once the epilogue warps have signalled
        for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
            const uint32_t x = kOX + (odd ? sbuf_bytes(128, 16) : 0u);
#pragma unroll
            for (int round = 0; round < 8 && ok; ++round) {
                ok = warp_agree(mbar_wait(c.ready + (round & 1), (uint32_t)(round >> 1) & 1u));
                fence_after();
                if (ok) issue(c, round, !any, x);
                __syncwarp();
            }
            any = true;
            odd = !odd;
        }
        // nothing of ours may still be running when TMEM is read for the flush, or freed
        if (elect_one()) commit(fin);
        ok = mbar_wait(fin, 0) && ok;
        any = false;                             // no rows to flush
    }
    for (int t = blockIdx.x; warp < kEpiWarps && t < a.ntiles && ok; t += gridDim.x) {
        any = true;
        const uint32_t x = kOX + (odd ? sbuf_bytes(128, 16) : 0u);
        odd = !odd;
        const int g = t * 128 + c.row;
        const bool valid = g < a.n;
        const bool p0 = c.part == 0;             // warpgroup 0: the row's inputs, X and the loss
        // this row's s_G, u and current d_feat, loaded now so that the forward rounds hide their latency
        float fg[kS], df[kS], ug = 0.f;
        if (valid && p0) {
            const float4 f0 = reinterpret_cast<const float4*>(a.feat)[2 * (size_t)g];
            const float4 f1 = reinterpret_cast<const float4*>(a.feat)[2 * (size_t)g + 1];
            fg[0] = f0.x; fg[1] = f0.y; fg[2] = f0.z; fg[3] = f0.w;
            fg[4] = f1.x; fg[5] = f1.y; fg[6] = f1.z; fg[7] = f1.w;
            ug = a.unc[g];
#pragma unroll
            for (int k = 0; k < kS; ++k) df[k] = a.d_feat[(size_t)g * a.d_feat_stride + k];
        } else {
#pragma unroll
            for (int k = 0; k < kS; ++k) fg[k] = df[k] = 0.f;
        }
        if (p0) {   // X = [p, 1, 0...]
            float v[8] = {0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 0.f}, z[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (valid) {
                v[0] = a.means[3 * (size_t)g];
                v[1] = a.means[3 * (size_t)g + 1];
                v[2] = a.means[3 * (size_t)g + 2];
            }
            sbuf_store8(SBuf{c.sm + x, 16}, c.row, 0, v);
            sbuf_store8(SBuf{c.sm + x, 16}, c.row, 8, z);
        }
        if (!(ok = next_round(c, 0))) break;
        hidden_epilogue(c, b1, kOH1);
        if (!(ok = next_round(c, 1))) break;
        hidden_epilogue(c, b2, kOH2);
        if (!(ok = next_round(c, 2))) break;
        hidden_epilogue(c, b3, kOH3);
        if (!(ok = next_round(c, 3))) break;
        if (p0) {   // loss and the output gradient
            float z[16];
            tmem_ld16(c.tmem + c.lanef + kAcc, z);
            float diff[kS], nn = 0.f;
#pragma unroll
            for (int k = 0; k < kS; ++k) {
                const float s = z[k] + b4[k];
                if (valid && a.s_mlp) a.s_mlp[(size_t)g * kS + k] = s;
                diff[k] = valid ? s - fg[k] : 0.f;
                nn = fmaf(diff[k], diff[k], nn);
            }
            nn = sqrtf(nn);
            const float wgt = valid ? fmaxf(ug, a.w_s) : 0.f;
            lsum += (double)((1.f + wgt) * nn);
            const float inv = nn > 0.f ? a.scale / nn : 0.f;
            float dz[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) dz[k] = k < kS ? diff[k] * inv : 0.f;
            if (valid)
#pragma unroll
                for (int k = 0; k < kS; ++k) a.d_feat[(size_t)g * a.d_feat_stride + k] = df[k] - wgt * dz[k];
            sbuf_store8(SBuf{c.sm + kODZ, 16}, c.row, 0, dz);
            sbuf_store8(SBuf{c.sm + kODZ, 16}, c.row, 8, dz + 8);
            db4acc += colsum16(dz, lane);       // lanes 2k, 2k+1: column k (k < 8)
        }
        if (!(ok = next_round(c, 4))) break;
        grad_epilogue(c, kOH3, kOD);         // dH3
        if (!(ok = next_round(c, 5))) break;
        grad_epilogue(c, kOH2, kOH3);        // dH2 over H3 (read by dW4, complete)
        if (!(ok = next_round(c, 6))) break;
        grad_epilogue(c, kOH1, kOD);         // dH1 over dH3 (read by dW3, complete)
        // dW1: nothing here waits for it
        fence_proxy_async();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(c.ready + 1);
    }
    if (warp < kEpiWarps) ok = warp_agree(mbar_wait(fin, 0)) && ok;
    fence_after();
    ok = !__syncthreads_or(!ok);
    if (!ok) {
        if (threadIdx.x == 0) atomicExch(&g_smooth_error, 1);
    } else if (any) {
        // flush: TMEM lane = this thread's row of each accumulator; warpgroup p takes
        // columns [32 p, 32 p + 32) of dW2 and dW3 and one of the small blocks
        float v[16];
        const int r = c.row;
#pragma unroll
        for (int q = 2 * c.part; q < 2 * c.part + 2; ++q) {
            tmem_ld16(c.tmem + c.lanef + kDW2 + 16 * q, v);
            red_row<16>(a.dW2 + (size_t)r * kH + 16 * q, v, 1.f, red_vec(a.dW2));
            tmem_ld16(c.tmem + c.lanef + kDW3 + 16 * q, v);
            red_row<16>(a.dW3 + (size_t)r * kH + 16 * q, v, 1.f, red_vec(a.dW3));
        }
        if (c.part == 0) {
            tmem_ld16(c.tmem + c.lanef + kDW1, v);
#pragma unroll
            for (int j = 0; j < 3; ++j) atomicAdd(a.dW1 + (size_t)r * 3 + j, v[j]);
            atomicAdd(a.db1 + r, v[3]);
        } else if (c.part == 1) {
            tmem_ld16(c.tmem + c.lanef + kDW4, v);    // row r = h3 dim, column k = output k
#pragma unroll
            for (int k = 0; k < kS; ++k) atomicAdd(a.dW4 + (size_t)k * kH + r, v[k]);
        } else if (c.part == 2) {
            tmem_ld16(c.tmem + c.lanef + kDB2, v);
            atomicAdd(a.db2 + r, v[0]);
        } else {
            tmem_ld16(c.tmem + c.lanef + kDB3, v);
            atomicAdd(a.db3 + r, v[0]);
        }
        if (c.part == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
            // one FP32 add per CTA: the order of several hundred showed in the loss at 1e-6
            double* const part = reinterpret_cast<double*>(c.sm + kODZ);
            if (lane == 0) part[warp] = lsum;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (threadIdx.x == 0)
                atomicAdd(a.loss, (float)((part[0] + part[1] + part[2] + part[3]) * (double)a.scale));
            if ((lane & 1) == 0 && (lane >> 1) < kS) atomicAdd(a.db4 + (lane >> 1), db4acc);
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(c.tmem, 512);
}

}  // namespace

// Reads and clears the smoothing kernel's timeout record.
le_status smooth_take_timeout(bool* timed_out)
{
    int flag = 0;
    LE_CUDA(cudaMemcpyFromSymbol(&flag, g_smooth_error, sizeof(int)));
    if (flag) {
        const int zero = 0;
        LE_CUDA(cudaMemcpyToSymbol(g_smooth_error, &zero, sizeof(int)));
    }
    *timed_out = flag != 0;
    return LE_OK;
}

}  // namespace leg

using namespace leg;

extern "C" le_status le_smooth(int32_t n, const float* means, const float* feat, const float* unc,
                               const le_smooth_mlp* mlp, float w_s, float lambda_smo, float* loss, float* d_feat,
                               int32_t d_feat_stride, const le_smooth_mlp_grads* dmlp, float* s_mlp, void* stream)
{
    LE_TRACE("le_smooth");
    LE_CHECK_ARG(n >= 0, "n = %d < 0", n);
    LE_CHECK_ARG(mlp && dmlp && loss, "null mlp / gradient / loss pointer");
    LE_CHECK_ARG(mlp->W1 && mlp->b1 && mlp->W2 && mlp->b2 && mlp->W3 && mlp->b3 && mlp->W4 && mlp->b4,
                 "null MLP parameter");
    LE_CHECK_ARG(dmlp->W1 && dmlp->b1 && dmlp->W2 && dmlp->b2 && dmlp->W3 && dmlp->b3 && dmlp->W4 && dmlp->b4,
                 "null MLP gradient");
    LE_CHECK_ARG(n == 0 || (means && feat && unc && d_feat), "null per-Gaussian pointer");
    LE_CHECK_ARG(d_feat_stride >= 8, "d_feat_stride = %d < 8", d_feat_stride);
    LE_CHECK_ARG(n == 0 || aligned16(feat), "feat must be 16-byte aligned");
    cudaStream_t s = as_stream(stream);
    const tc::ZeroList zl{{loss, dmlp->W1, dmlp->b1, dmlp->W2, dmlp->b2, dmlp->W3, dmlp->b3, dmlp->W4, dmlp->b4},
                          {1, kH * 3, kH, kH * kH, kH, kH * kH, kH, kS * kH, kS}};
    const le_status zs = tc::zero_list(zl, 9, s);
    if (zs != LE_OK) return zs;
    if (n == 0) return LE_OK;
    int dev = 0, sms = 0;
    LE_CUDA(cudaGetDevice(&dev));
    LE_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SmoothArgs a;
    a.n = n;
    a.ntiles = (n + 127) / 128;
    a.means = means;
    a.feat = feat;
    a.unc = unc;
    a.W1 = mlp->W1;
    a.b1 = mlp->b1;
    a.W2 = mlp->W2;
    a.b2 = mlp->b2;
    a.W3 = mlp->W3;
    a.b3 = mlp->b3;
    a.W4 = mlp->W4;
    a.b4 = mlp->b4;
    a.w_s = w_s;
    a.scale = lambda_smo / (float)n;
    a.loss = loss;
    a.d_feat = d_feat;
    a.d_feat_stride = d_feat_stride;
    a.s_mlp = s_mlp;
    a.dW1 = dmlp->W1;
    a.db1 = dmlp->b1;
    a.dW2 = dmlp->W2;
    a.db2 = dmlp->b2;
    a.dW3 = dmlp->W3;
    a.db3 = dmlp->b3;
    a.dW4 = dmlp->W4;
    a.db4 = dmlp->b4;
    LE_CUDA(cudaFuncSetAttribute(smooth_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmoothSmem));
    const int grid = a.ntiles < sms ? a.ntiles : sms;
    smooth_kernel<<<grid, kThreadsS, kSmoothSmem, s>>>(a);
    LE_LAUNCHED();
    return LE_OK;
}
