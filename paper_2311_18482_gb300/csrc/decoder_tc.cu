// Fused semantic decoder on the 5th-generation tensor cores (tcgen05, BF16
// operands, FP32 accumulation in TMEM).
//
// D_MLP (Eq. 8, eq:lem_dec; supp. Tab. dmlp, here 8 -> 64 -> 128 -> N) runs per
// 128-pixel tile: the rendered feature R_s of the tile is the A operand of
// three chained MMAs whose accumulators never leave the SM; the CUDA cores
// only apply bias + ReLU between layers (TMEM -> registers -> BF16 shared
// memory) and the softmax at the end.  Four kernels share that front end:
//
//   dec_fwd_kernel    inference (supp. Sec. "Inference"): argmax and/or
//                     M_infer = softmax(logits), four tiles in flight per CTA
//                     (two above 128 codes).
//   dec_train_kernel  training step (Eqs. 9-12): uncertainty-weighted CE,
//                     dL/dR_u, and the whole backward on the tensor cores,
//                     warp-specialised with two tiles in flight (one MMA
//                     warp, four epilogue warpgroups).  dL/dz, dL/dh2 and
//                     dL/dh1 are written once, pixel-major; the input-gradient
//                     MMAs read them K-major and the weight-gradient MMAs read
//                     the same buffers MN-major (contracting over the tile's
//                     pixels); bias gradients are MMAs against a ones operand.
//                     Weight gradients accumulate in TMEM over all tiles of a
//                     CTA and are flushed once.
//   query_fused_kernel relevancy (supp. Sec. "Inference", LERF): with
//                     p proportional to e = exp(z - max z), |F_clip|^2 =
//                     p^T (S_c S_c^T) p and phi.q_j = p.(S_c q_j)/|F_clip|; the
//                     relevancy does not depend on the scale of p, so neither
//                     the softmax normaliser nor the 896-dim feature map F is
//                     ever formed.
//   export_fused_kernel the feature map F itself, where a consumer wants it.
//
// Every mbarrier wait is bounded (about a second); on timeout the kernel
// records it in g_tc_error, stops issuing work, frees its TMEM and returns.
#include "tc_common.cuh"

namespace leg {

__device__ int g_tc_error;

namespace {
using namespace tc;

constexpr int kD = 8, kH1 = 64, kH2 = 128;

struct DecArgs {
    int P, ncb;
    const float *feat, *unc;
    const int32_t* target;
    const float *W1, *b1, *W2, *b2, *W3, *b3;
    float lambda_ce, lambda_u, invP;
    float* loss;
    float *d_feat, *d_unc;
    float *dW1, *db1, *dW2, *db2, *dW3, *db3;
    int32_t* argmax;
    float* prob;
    // query and feature-map export: the back phase's operand, a chunked BF16 image
    // (query_prep_kernel, codebook_chunks_kernel) of `dd` rows or dims
    const unsigned char* G_img;
    int dd;
    // query
    int Q, n_neg;
    float* rel;
    // training with the RGB L1 term of the same pixels (nullable img): img, img_t [3, P],
    // d_img [3, P] = sign(img - img_t) inv_l1, *loss_l1 += sum |img - img_t| inv_l1
    const float *img, *img_t;
    float *d_img, *loss_l1;
    float inv_l1;
};

// Per-warpgroup state of the shared MLP front end.  With nhalf = 2, two
// warpgroups serve the same 128 TMEM lanes (rows) and split every epilogue by
// columns; `xch` is their shared-memory exchange for row-wide statistics.
struct Front {
    SBuf W1s, W2s, W3s, X1, H1, H2;
    const float *b1s, *b2s, *b3s;
    uint64_t* mbar;
    uint32_t phase;
    uint32_t tw;       // TMEM column base of this warpgroup's working accumulator
    uint32_t lane;     // this warp's TMEM lane field
    int tid;           // row of the tile (TMEM lane) this thread serves
    int bar_id, nthreads;
    bool issuer;       // the warp that issues this group's MMAs (warp-uniform)
    int half, nhalf;
    float4* xch;       // [2][128] (nhalf = 2 only)
};

// Columns [c0, c1) of an N-column epilogue handled by this thread's half (units of 16).
__device__ __forceinline__ void my_cols(const Front& f, int N, int& c0, int& c1)
{
    const int nch = N / 16, per = (nch + f.nhalf - 1) / f.nhalf;
    c0 = min(nch, f.half * per) * 16;
    c1 = min(nch, (f.half + 1) * per) * 16;
}

__device__ __forceinline__ void wg_sync(const Front& f)
{
    asm volatile("bar.sync %0, %1;" ::"r"(f.bar_id), "r"(f.nthreads) : "memory");
}

// Wait for this warpgroup's MMA barrier; false (for every thread) if any thread timed out.
__device__ __forceinline__ bool wg_wait(Front& f)
{
    const bool ok = mbar_wait(f.mbar, f.phase);
    f.phase ^= 1u;
    const bool bad = bar_any(f.bar_id, f.nthreads, !ok);
    if (bad && f.tid == 0) atomicExch(&g_tc_error, 1);
    fence_after();
    return !bad;
}

// Make this warpgroup's shared-memory writes visible to the tensor core and
// order them (and all TMEM reads) before the MMAs issued next.
__device__ __forceinline__ void wg_publish(const Front& f)
{
    fence_proxy_async();
    fence_before();
    wg_sync(f);
    fence_after();
}

// R_s of pixel p (zeros past the end), for mlp_forward_x.
__device__ __forceinline__ void load_feat(const DecArgs& a, int p, bool valid, float* x)
{
#pragma unroll
    for (int c = 0; c < 8; ++c) x[c] = valid ? a.feat[(size_t)c * a.P + p] : 0.f;
}

// D_MLP forward of one 128-pixel tile: X1 <- x (col 8 = 1 for the bias
// gradient), H1 = relu(W1 x + b1), H2 = relu(W2 h1 + b2), logits - b3 left in
// TMEM columns [tw, tw + ncb).  The tile's features come in registers (x, read
// by the first part only), so that a caller can load them a tile ahead.
// Returns false on a timed-out wait.
__device__ bool mlp_forward_x(Front& f, const DecArgs& a, const float* x)
{
    float v[16];
    uint32_t w[8];
    if (f.half == 0) sbuf_store8(f.X1, f.tid, 0, x);
    if (f.half == f.nhalf - 1) {
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = c == 0 ? 1.f : 0.f;
        sbuf_store8(f.X1, f.tid, 8, v);
    }
    wg_publish(f);
    if (f.issuer && elect_one()) {
        mma(f.tw, kdesc(f.X1, 0, 0), kdesc(f.W1s, 0, 0), idesc_bf16(kH1, false, false), 0);
        commit(f.mbar);
    }
    if (!wg_wait(f)) return false;
    int c0, c1;
    my_cols(f, kH1, c0, c1);
    for (int c = c0; c < c1; c += 16) {
        tmem_ld16(f.tw + f.lane + c, v);
        relu16(v, f.b1s + c, w);
        sts_row16(smem_u32(f.H1.p) + sbuf_off(f.tid, c, f.H1.C), w);
    }
    wg_publish(f);
    if (f.issuer && elect_one()) {
#pragma unroll
        for (int s = 0; s < kH1 / 16; ++s)
            mma(f.tw, kdesc(f.H1, 0, 16 * s), kdesc(f.W2s, 0, 16 * s), idesc_bf16(kH2, false, false), s > 0);
        commit(f.mbar);
    }
    if (!wg_wait(f)) return false;
    my_cols(f, kH2, c0, c1);
    for (int c = c0; c < c1; c += 16) {
        tmem_ld16(f.tw + f.lane + c, v);
        relu16(v, f.b2s + c, w);
        sts_row16(smem_u32(f.H2.p) + sbuf_off(f.tid, c, f.H2.C), w);
    }
    wg_publish(f);
    if (f.issuer && elect_one()) {
        const uint32_t id = idesc_bf16(a.ncb, false, false);
#pragma unroll
        for (int s = 0; s < kH2 / 16; ++s)
            mma(f.tw, kdesc(f.H2, 0, 16 * s), kdesc(f.W3s, 0, 16 * s), id, s > 0);
        commit(f.mbar);
    }
    return wg_wait(f);
}

// Online max / argmax / log-sum-exp over the ncb logits in TMEM (+ b3), ties to
// the lowest index.  Without a branch per column: a new maximum (s e + 1) and a
// smaller logit (s 1 + e) are one FMA of selected factors, e = exp(-|z - max|).
__device__ __forceinline__ void logits_lse(const Front& f, int ncb, float& lse, int& am)
{
    float m = -INFINITY, s = 0.f, v[16];
    am = 0;
    for (int c = 0; c < ncb; c += 16) {
        tmem_ld16(f.tw + f.lane + c, v);
        add_bias16(v, f.b3s + c);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float z = v[j];
            const bool up = z > m;
            const float e = __expf(-fabsf(z - m));
            s = __fmaf_rn(s, up ? e : 1.f, up ? 1.f : e);
            m = up ? z : m;
            am = up ? c + j : am;
        }
    }
    lse = m + __logf(s);
}

__host__ __device__ constexpr size_t weights_bytes(int ncb)
{
    return (size_t)sbuf_bytes(64, 16) + sbuf_bytes(128, 64) + sbuf_bytes(ncb, 128) +
           ((size_t)(64 + 128 + ncb) * 4 + 127) / 128 * 128;
}

// Carve weights + biases at `base`, fill them (all threads).
__device__ unsigned char* load_weights(unsigned char* base, const DecArgs& a, Front& f)
{
    unsigned char* p = base;
    f.W1s = SBuf{p, 16};
    p += sbuf_bytes(64, 16);
    f.W2s = SBuf{p, 64};
    p += sbuf_bytes(128, 64);
    f.W3s = SBuf{p, 128};
    p += sbuf_bytes(a.ncb, 128);
    float* bs = reinterpret_cast<float*>(p);
    p += ((size_t)(64 + 128 + a.ncb) * 4 + 127) / 128 * 128;
    sbuf_fill(f.W1s, 64, a.W1, kD, 64, kD);
    sbuf_fill_rows(f.W2s, 128, a.W2);
    sbuf_fill_rows(f.W3s, a.ncb, a.W3);
    for (int i = threadIdx.x; i < 64 + 128 + a.ncb; i += blockDim.x)
        bs[i] = i < 64 ? a.b1[i] : (i < 192 ? a.b2[i - 64] : a.b3[i - 192]);
    f.b1s = bs;
    f.b2s = bs + 64;
    f.b3s = bs + 192;
    return p;
}

// ---------------------------------------------------------------------------
// Inference.  NWG warpgroups per CTA, each with its own tile, buffers, mbarrier
// and 512 / NWG TMEM columns; weights shared.  A tile is a chain of three MMA
// rounds and their epilogues, so the tiles in flight per SM set the rate: four
// up to 128 codes (H2 takes the place of X1 and H1, which have been read by
// then), two above, where a tile's logits need 256 columns.  Tiles are dealt out
// over the CTAs first, so a small image spreads over the SMs.  With two tiles of
// 128 codes in flight and a branch per logit in the softmax, 10,000 / 300,000 /
// 1,088,640 pixels took 19.8 / 114 / 370 us at 128 codes and 31.8 / 194 / 629 us
// at 256; now 10.3 / 52 / 157 us and 14.7 / 100 / 322 us.
constexpr size_t kFwdTileBytes = sbuf_bytes(128, 128);

__host__ constexpr size_t fwd_smem(int ncb, int nwg) { return weights_bytes(ncb) + nwg * kFwdTileBytes + 128; }

template <int NWG>
__global__ void __launch_bounds__(128 * NWG, 1) dec_fwd_kernel(DecArgs a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    constexpr int kCols = 512 / NWG;
    Front f;
    unsigned char* p = load_weights(sm, a, f);
    const int warp = (int)warp_uniform(threadIdx.x >> 5), wg = warp >> 2;
    unsigned char* q = p + wg * kFwdTileBytes;
    f.X1 = SBuf{q, 16};
    f.H1 = SBuf{q + sbuf_bytes(128, 16), 64};
    f.H2 = SBuf{q, 128};
    uint64_t* mbars = reinterpret_cast<uint64_t*>(p + NWG * kFwdTileBytes);
    uint32_t* slot = reinterpret_cast<uint32_t*>(mbars + NWG);
    f.mbar = mbars + wg;
    f.phase = 0;
    f.tid = threadIdx.x & 127;
    f.bar_id = 1 + wg;
    f.issuer = (warp & 3) == 0;
    f.nthreads = 128;
    f.half = 0;
    f.nhalf = 1;
    f.xch = nullptr;
    if (threadIdx.x == 0)
        for (int w = 0; w < NWG; ++w) mbar_init(mbars + w, 1);
    if (threadIdx.x < 32) tmem_alloc(slot, 512);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tbase = warp_uniform(*reinterpret_cast<volatile uint32_t*>(slot));
    f.tw = tbase + kCols * wg;
    f.lane = (uint32_t)(32 * (f.tid >> 5)) << 16;

    const int ntiles = (a.P + 127) / 128;
    const auto tile_px = [&](int tile) { return tile < ntiles ? tile * 128 + f.tid : a.P; };
    float x[8];                                 // this tile's R_s, loaded a tile ahead
    int tile = blockIdx.x + gridDim.x * wg;
    load_feat(a, tile_px(tile), tile_px(tile) < a.P, x);
    for (; tile < ntiles; tile += gridDim.x * NWG) {
        const int px = tile * 128 + f.tid;
        const bool valid = px < a.P;
        if (!mlp_forward_x(f, a, x)) break;
        const int nx = tile_px(tile + (int)gridDim.x * NWG);
        load_feat(a, nx, nx < a.P, x);
        float lse;
        int am;
        logits_lse(f, a.ncb, lse, am);
        if (valid && a.argmax) a.argmax[px] = am;
        if (a.prob) {
            float v[16];
            for (int c = 0; c < a.ncb; c += 16) {
                tmem_ld16(f.tw + f.lane + c, v);
                add_bias16(v, f.b3s + c);
                if (valid)
#pragma unroll
                    for (int j = 0; j < 16; ++j) a.prob[(size_t)(c + j) * a.P + px] = __expf(v[j] - lse);
            }
        }
        fence_before();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (threadIdx.x < 32) tmem_dealloc(tbase, 512);
}

// ---------------------------------------------------------------------------
// Training.  One CTA per SM, persistent over tiles and warp-specialised: warp
// 16 issues every MMA; warpgroups 0-3 run the epilogues of two tiles in flight
// (slot s = warpgroups 2s and 2s+1, which serve the same 128 rows and split
// every epilogue by columns), so the tensor core works on one slot while the
// CUDA cores finish the other.  Per tile, six MMA stages alternate with six
// epilogues (z = logits, dz = dL/dz etc.):
//   S1  h1 = X1 W1^T                                E1  bias, ReLU -> H1
//   S2  h2 = H1 W2^T                                E2  bias, ReLU -> H2
//   S3  z  = H2 W3^T                                E3  softmax, CE (Eqs. 9-12) -> dz into D
//   S4  dh2 = dz W3;  dW3 += dz^T h2;  db3 += dz^T 1   E4  mask (h2 > 0) -> dh2 into H2's buffer
//   S5  dh1 = dh2 W2; dW2 += dh2^T h1; db2 += dh2^T 1  E5  mask (h1 > 0) -> dh1 into D
//   S6  dx  = dh1 W1; [dW1 | db1] += dh1^T [x | 1]     E6  dx -> d_feat
// dz, dh2 and dh1 are stored pixel-major: the input-gradient MMAs read them
// K-major and the weight-gradient MMAs MN-major (contracting over the tile's
// pixels).  Handshake per slot: its eight epilogue warps arrive on ready[s]
// once their operand is in shared memory and their TMEM reads are done; the
// MMA thread waits, issues, and commits to done[s].  All MMAs come from one
// thread, so the weight-gradient accumulations of both slots are ordered.
// TMEM (512 columns): working accumulators [0,128) and [128,256); dW3
// [256,384); dW2 [384,448); block P [448,464) holds db2 (column 0, again in 9)
// and db3 (column 8); block Q [480,496) holds dW1 (columns 0-7) and db1 (8).
// The ones operand E (128 pixels x 24, ones in columns 8 and 17) read from
// column 0 sums over pixels into output column 8, read from column 8 into
// columns 0 and 9 -- so db3 and db2 share block P without overlapping.
constexpr int kTrainThreads = 4 * 128 + 32;
constexpr uint32_t kTW3 = 256, kTW2 = 384, kTP = 448, kTQ = 480;
constexpr int kEC = 24;

// Shared-memory addresses of one slot's buffers (column counts 16, 64, 128, 128):
// X1; H1; H2, later dh2; D: dz (and the softmax exchange), later dh1.
constexpr uint32_t kSX1 = 0, kSH1 = sbuf_bytes(128, 16), kSH2 = kSH1 + sbuf_bytes(128, kH1),
                   kSD = kSH2 + sbuf_bytes(128, 128), kSlotBytes = kSD + sbuf_bytes(128, 128);

__host__ __device__ constexpr size_t train_slot_bytes() { return kSlotBytes; }

__host__ constexpr size_t train_smem(int ncb)
{
    return weights_bytes(ncb) + sbuf_bytes(128, kEC) + 2 * train_slot_bytes() + 128;
}

// Issue MMA stage `st` (0-5) of the slot whose buffers start at shared address
// q.  `init`: the first tile of this CTA, whose weight-gradient MMAs overwrite
// their accumulators.  Each operand's descriptor is built once per stage; the
// next 16-wide K step only moves the start address, by 16 (K-major: one pair
// of core matrices, 256 B) or by 2C (MN-major over a C-column buffer: two
// 8-row groups, 32 C bytes) in descriptor units of 16 B.
__device__ __forceinline__ void train_stage(int st, int ncb, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t e,
                                            uint32_t q, uint32_t tw, uint32_t tb, bool init)
{
    const uint32_t keep = init ? 0u : 1u;
    const uint32_t x1 = q + kSX1, h1 = q + kSH1, h2 = q + kSH2, d = q + kSD;
    switch (st) {
        case 0:
            mma(tw, kdesc_at(x1, 16, 0, 0), kdesc_at(w1, 16, 0, 0), idesc_bf16(kH1, false, false), 0);
            break;
        case 1: {
            const uint64_t a = kdesc_at(h1, kH1, 0, 0), b = kdesc_at(w2, kH1, 0, 0);
#pragma unroll
            for (int k = 0; k < kH1 / 16; ++k) mma(tw, a + 16 * k, b + 16 * k, idesc_bf16(kH2, false, false), k > 0);
            break;
        }
        case 2: {
            const uint64_t a = kdesc_at(h2, 128, 0, 0), b = kdesc_at(w3, 128, 0, 0);
            const uint32_t id = idesc_bf16(ncb, false, false);
#pragma unroll
            for (int k = 0; k < kH2 / 16; ++k) mma(tw, a + 16 * k, b + 16 * k, id, k > 0);
            break;
        }
        case 3: {
            const uint64_t ak = kdesc_at(d, 128, 0, 0), w3m = mndesc_at(w3, 128, 0, 0);
            for (int k = 0; k < ncb / 16; ++k)
                mma(tw, ak + 16 * k, w3m + 256 * k, idesc_bf16(kH2, false, true), k > 0);
            const uint64_t am = mndesc_at(d, 128, 0, 0), h2m = mndesc_at(h2, 128, 0, 0), em = mndesc_at(e, kEC, 0, 0);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(tb + kTW3, am + 256 * k, h2m + 256 * k, idesc_bf16(kH2, true, true), k > 0 ? 1u : keep);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(tb + kTP, am + 256 * k, em + 2 * kEC * k, idesc_bf16(16, true, true), k > 0 ? 1u : keep);
            break;
        }
        case 4: {
            const uint64_t ak = kdesc_at(h2, 128, 0, 0), w2m = mndesc_at(w2, kH1, 0, 0);
#pragma unroll
            for (int k = 0; k < kH2 / 16; ++k)
                mma(tw, ak + 16 * k, w2m + 2 * kH1 * k, idesc_bf16(kH1, false, true), k > 0);
            const uint64_t am = mndesc_at(h2, 128, 0, 0), h1m = mndesc_at(h1, kH1, 0, 0),
                           em = mndesc_at(e, kEC, 0, 8);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(tb + kTW2, am + 256 * k, h1m + 2 * kH1 * k, idesc_bf16(kH1, true, true), k > 0 ? 1u : keep);
#pragma unroll
            for (int k = 0; k < 8; ++k) mma(tb + kTP, am + 256 * k, em + 2 * kEC * k, idesc_bf16(16, true, true), 1u);
            break;
        }
        default: {
            const uint64_t ak = kdesc_at(d, 128, 0, 0), w1m = mndesc_at(w1, 16, 0, 0);
#pragma unroll
            for (int k = 0; k < kH1 / 16; ++k)
                mma(tw, ak + 16 * k, w1m + 2 * 16 * k, idesc_bf16(16, false, true), k > 0);
            const uint64_t am = mndesc_at(d, 128, 0, 0), x1m = mndesc_at(x1, 16, 0, 0);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                mma(tb + kTQ, am + 256 * k, x1m + 2 * 16 * k, idesc_bf16(16, true, true), k > 0 ? 1u : keep);
            break;
        }
    }
}

// The MMA warp: tile pairs in order, stage by stage, slot 0 then slot 1.
__device__ __forceinline__ bool train_mma_loop(int ncb, const Front& f, uint32_t e, uint32_t slots,
                                               uint64_t* ready, uint64_t* done, uint32_t tb, int ntiles)
{
    uint32_t ph[2] = {0u, 0u};
    const uint32_t w1 = smem_u32(f.W1s.p), w2 = smem_u32(f.W2s.p), w3 = smem_u32(f.W3s.p);
    for (int it = 0;; ++it) {
        const int t0 = blockIdx.x + 2 * it * gridDim.x;
        if (t0 >= ntiles) break;
        const int nsl = t0 + (int)gridDim.x < ntiles ? 2 : 1;
        for (int st = 0; st < 6; ++st)
            for (int s = 0; s < nsl; ++s) {
                if (!warp_agree(mbar_wait(ready + s, ph[s]))) return false;
                ph[s] ^= 1u;
                fence_after();
                if (elect_one()) {
                    train_stage(st, ncb, w1, w2, w3, e, slots + kSlotBytes * s, tb + 128u * s, tb, it == 0 && s == 0);
                    commit(done + s);
                }
                __syncwarp();
            }
    }
    return true;
}

// Epilogue thread state: slot s (buffers at shared address sb), half h of the
// columns, tile row `row`.
struct EpiCtx {
    uint32_t sb;
    uint64_t *ready, *done;
    uint32_t tw, lanef, ph;
    int s, h, row, bar_id;
};

__device__ __forceinline__ void epi_signal(const EpiCtx& e)
{
    fence_proxy_async();
    fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(e.ready);
}

// Wait for the slot's MMAs; the outcome is made uniform over the slot's 256
// threads, so a timeout never leaves part of them at the exchange barrier.
__device__ __forceinline__ bool epi_wait(EpiCtx& e)
{
    const bool ok = !bar_any(e.bar_id, 256, !mbar_wait(e.done, e.ph));
    e.ph ^= 1u;
    fence_after();
    return ok;
}

// Byte offset of exchange entry i (0-255) in the 128-column canonical buffer D:
// the 16-byte chunk (row 8 (i/16) + i%8, columns 8 ((i/8)%2) ...), i.e. every
// entry lies in columns [0, 16).
__device__ __forceinline__ uint32_t xch_off(int i)
{
    return (uint32_t)((i >> 4) * 2048 + ((i >> 3) & 1) * 128 + (i & 7) * 16);
}

// 16 columns [c, c + 16) of row `row` of the C-column buffer at shared address b.
__device__ __forceinline__ void store16(uint32_t b, int C, int row, int c, const float* v)
{
    sts_bf16x8(b + sbuf_off(row, c, C), v);
    sts_bf16x8(b + sbuf_off(row, c + 8, C), v + 8);
}

// v[idx] for a runtime idx in [0, 16), by a select tree over the index bits
// (keeps v in registers).
__device__ __forceinline__ float select16(const float* v, int idx)
{
    float t8[8], t4[4], t2[2];
    const bool b0 = idx & 1, b1 = idx & 2, b2 = idx & 4, b3 = idx & 8;
#pragma unroll
    for (int i = 0; i < 8; ++i) t8[i] = b0 ? v[2 * i + 1] : v[2 * i];
#pragma unroll
    for (int i = 0; i < 4; ++i) t4[i] = b1 ? t8[2 * i + 1] : t8[2 * i];
#pragma unroll
    for (int i = 0; i < 2; ++i) t2[i] = b2 ? t4[2 * i + 1] : t4[2 * i];
    return b3 ? t2[1] : t2[0];
}

__device__ __forceinline__ bool train_epilogue(const DecArgs& a, const float* bias, EpiCtx& e, int ntiles,
                                               float& acc_ce, float& acc_u, float& acc_l1)
{
    constexpr float kL2E = 1.4426950408889634f;
    const int row = e.row, h = e.h;
    const float *b1s = bias, *b2s = bias + kH1, *b3s = bias + kH1 + kH2;
    const uint32_t tl = e.tw + e.lanef;
    const int nu = a.ncb / 16, per = (nu + 1) / 2;
    const int c0 = min(nu, h * per) * 16, c1 = min(nu, (h + 1) * per) * 16;   // this half's logit columns
    float v[16];
    // this row's inputs of the slot's next tile, loaded one tile ahead so that
    // their latency is not on the path from one tile's first MMA to the next:
    // half 0 the feature, half 1 (with the L1 term) the image and its target
    float pf[8], pu = 0.f;
    int pt = -1;
    auto fetch = [&](int tile_n) {
        const int pxn = tile_n * 128 + row;
        const bool vn = tile_n < ntiles && pxn < a.P;
        if (h == 0) {
#pragma unroll
            for (int c = 0; c < 8; ++c) pf[c] = vn ? a.feat[(size_t)c * a.P + pxn] : 0.f;
        } else if (a.img) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                pf[c] = vn ? a.img[(size_t)c * a.P + pxn] : 0.f;
                pf[3 + c] = vn ? a.img_t[(size_t)c * a.P + pxn] : 0.f;
            }
        }
        pu = vn ? a.unc[pxn] : 0.f;
        pt = vn ? a.target[pxn] : -1;
    };
    fetch(blockIdx.x + e.s * gridDim.x);
    for (int it = 0;; ++it) {
        const int tile = blockIdx.x + (2 * it + e.s) * gridDim.x;
        if (tile >= ntiles) break;
        const int px = tile * 128 + row;
        const bool valid = px < a.P;
        const uint32_t sb = opaque(e.sb);
        const uint32_t X1 = sb + kSX1, H1 = sb + kSH1, H2 = sb + kSH2, D = sb + kSD;
        // X1 = [feat | 1 | 0]: the ones column gives db1
        if (h == 0) {
#pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = pf[c];
            sts_bf16x8(X1 + sbuf_off(row, 0, 16), v);
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = c == 0 ? 1.f : 0.f;
            sts_bf16x8(X1 + sbuf_off(row, 8, 16), v);
            if (a.img && valid) {
                // the RGB L1 term of this pixel (the same operations as le_rgb_l1)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float r = pf[c] - pf[3 + c];
                    acc_l1 += fabsf(r);
                    a.d_img[(size_t)c * a.P + px] = r > 0.f ? a.inv_l1 : (r < 0.f ? -a.inv_l1 : 0.f);
                }
            }
        }
        const float u = pu;
        const int t = pt;
        fetch(tile + 2 * (int)gridDim.x);
        epi_signal(e);
        if (!epi_wait(e)) return false;
        // E1: h1 columns [32h, 32h + 32)
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            tmem_ld16(tl + 32 * h + 16 * k, v);
            relu16(v, b1s + 32 * h + 16 * k, w);
            sts_row16(H1 + sbuf_off(row, 32 * h + 16 * k, kH1), w);
        }
        epi_signal(e);
        if (!epi_wait(e)) return false;
        // E2: h2 columns [64h, 64h + 64)
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            tmem_ld16(tl + 64 * h + 16 * k, v);
            relu16(v, b2s + 64 * h + 16 * k, w);
            sts_row16(H2 + sbuf_off(row, 64 * h + 16 * k, 128), w);
        }
        epi_signal(e);
        if (!epi_wait(e)) return false;
        // E3: softmax over this half's logit columns [c0, c1).  Pass 1: max (and
        // the target's logit); pass 2: e = exp(z - max), their sum, e parked in
        // the free TMEM columns; exchange with the other half; pass 3: dz.
        const int jt = t - c0;
        const bool own_t = jt >= 0 && t < c1;
        float mh = -INFINITY, zt_h = 0.f;
#pragma unroll 1
        for (int uu = 0; uu < 4; ++uu)
            if (c0 + 16 * uu < c1) {
                tmem_ld16(tl + c0 + 16 * uu, v);
                add_bias16(v, b3s + c0 + 16 * uu);
#pragma unroll
                for (int j = 0; j < 16; ++j) mh = fmaxf(mh, v[j]);
                if (own_t && (jt >> 4) == uu) zt_h = select16(v, jt & 15);
            }
        const float mhl = mh * kL2E;
        float sh = 0.f;
#pragma unroll 1
        for (int uu = 0; uu < 4; ++uu)
            if (c0 + 16 * uu < c1) {
                tmem_ld16(tl + c0 + 16 * uu, v);
                add_bias16(v, b3s + c0 + 16 * uu);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    v[j] = ex2_approx(fmaf(v[j], kL2E, -mhl));
                    sh += v[j];
                }
                tmem_st16(tl + c0 + 16 * uu, v);
            }
        tmem_wait_st();
        // the halves exchange (max, sum, target logit) through D's columns [0, 16),
        // which pass 3 then overwrites with dz: no stale FP32 bits stay in D to
        // reach an MMA (as bf16 they can be Inf or NaN)
        float4 o;
        asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(D + xch_off(h * 128 + row)), "f"(mh), "f"(sh),
                     "f"(zt_h), "f"(0.f)
                     : "memory");
        asm volatile("bar.sync %0, 256;" ::"r"(e.bar_id) : "memory");
        asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                     : "=f"(o.x), "=f"(o.y), "=f"(o.z), "=f"(o.w)
                     : "r"(D + xch_off((1 - h) * 128 + row))
                     : "memory");
        asm volatile("bar.sync %0, 256;" ::"r"(e.bar_id) : "memory");
        const float m = fmaxf(mh, o.x);
        const float ssum = (c0 < c1 ? sh * ex2_approx((mh - m) * kL2E) : 0.f) +
                           (o.y > 0.f ? o.y * ex2_approx((o.x - m) * kL2E) : 0.f);
        const float lse = m + __logf(ssum);
        const float zt = own_t ? zt_h : o.z;
        const float ce = lse - zt;
        const float wce = valid ? a.lambda_ce * (1.f - u) : 0.f;
        if (valid && h == 0) {
            a.d_unc[px] = (a.lambda_u - a.lambda_ce * ce) * a.invP;
            acc_ce += ce * (1.f - u);
            acc_u += u;
        }
        // dz * P (1/P is applied when the gradients are written)
        const float scale = c0 < c1 ? wce * ex2_approx((mh - m) * kL2E) / ssum : 0.f;
#pragma unroll 1
        for (int uu = 0; uu < 4; ++uu)
            if (c0 + 16 * uu < c1) {
                tmem_ld16(tl + c0 + 16 * uu, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] *= scale;
                store16(D, 128, row, c0 + 16 * uu, v);
            }
        if (own_t && valid) {
            const float et = ex2_approx(fmaf(zt_h, kL2E, -mhl));
            const __nv_bfloat16 bv = __float2bfloat16_rn(et * scale - wce);
            asm volatile("st.shared.b16 [%0], %1;" ::"r"(D + sbuf_off(row, t, 128)),
                         "h"(*reinterpret_cast<const unsigned short*>(&bv))
                         : "memory");
        }
        epi_signal(e);
        if (!epi_wait(e)) return false;
        // E4: dh2 = (dz W3) * [h2 > 0] into H2's buffer
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            tmem_ld16(tl + 64 * h + 16 * k, v);
            const uint32_t at = H2 + sbuf_off(row, 64 * h + 16 * k, 128);
            relu_mask16(v, at, w);
            sts_row16(at, w);
        }
        epi_signal(e);
        if (!epi_wait(e)) return false;
        // E5: dh1 = (dh2 W2) * [h1 > 0] into D
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            tmem_ld16(tl + 32 * h + 16 * k, v);
            relu_mask16(v, H1 + sbuf_off(row, 32 * h + 16 * k, kH1), w);
            sts_row16(D + sbuf_off(row, 32 * h + 16 * k, 128), w);
        }
        epi_signal(e);
        if (!epi_wait(e)) return false;
        // E6: dx = dh1 W1 -> d_feat
        if (h == 0) {
            tmem_ld16(tl, v);
            if (valid)
#pragma unroll
                for (int c = 0; c < kD; ++c) a.d_feat[(size_t)c * a.P + px] = v[c] * a.invP;
        }
    }
    return true;
}

__global__ void __launch_bounds__(kTrainThreads, 1) dec_train_kernel(DecArgs a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    Front f;
    unsigned char* p = load_weights(sm, a, f);
    const SBuf E{p, kEC};
    p += sbuf_bytes(128, kEC);
    unsigned char* slots = p;
    const uint32_t slots_a = smem_u32(slots);
    p += 2 * train_slot_bytes();
    uint64_t* ready = reinterpret_cast<uint64_t*>(p);
    uint64_t* done = ready + 2;
    uint64_t* fin = ready + 4;
    uint32_t* slot_addr = reinterpret_cast<uint32_t*>(ready + 5);
    const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    // the slots start zeroed (padding columns feed MMA rows that are never read,
    // and must hold finite values); E has ones in columns 8 and 17
    for (size_t i = threadIdx.x; i < 2 * train_slot_bytes() / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(slots)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = threadIdx.x; i < 128 * (kEC / 8); i += blockDim.x) {
        const int r = i / (kEC / 8), cb = i % (kEC / 8);
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (cb == 1) v[0] = 1.f;
        if (cb == 2) v[1] = 1.f;
        sbuf_store8(E, r, 8 * cb, v);
    }
    if (threadIdx.x == 0) {
        mbar_init(ready, 8);
        mbar_init(ready + 1, 8);
        mbar_init(done, 1);
        mbar_init(done + 1, 1);
        mbar_init(fin, 1);
    }
    if (warp == 0) tmem_alloc(slot_addr, 512);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tb = warp_uniform(*reinterpret_cast<volatile uint32_t*>(slot_addr));
    const int ntiles = (a.P + 127) / 128;
    bool ok = true;
    float acc_ce = 0.f, acc_u = 0.f, acc_l1 = 0.f;
    if (warp == 16) {
        ok = train_mma_loop(a.ncb, f, smem_u32(E.p), slots_a, ready, done, tb, ntiles);
        if (ok) {
            if (elect_one()) commit(fin);
            ok = mbar_wait(fin, 0);
        }
    } else {
        EpiCtx e;
        e.s = warp >> 3;
        e.h = (warp >> 2) & 1;
        e.row = threadIdx.x & 127;
        e.sb = slots_a + kSlotBytes * e.s;
        e.ready = ready + e.s;
        e.done = done + e.s;
        e.tw = tb + 128u * e.s;
        e.lanef = (uint32_t)(32 * (warp & 3)) << 16;
        e.ph = 0;
        e.bar_id = 1 + e.s;
        ok = train_epilogue(a, f.b1s, e, ntiles, acc_ce, acc_u, acc_l1);
    }
    fence_before();
    const bool bad = __syncthreads_or(!ok);
    fence_after();
    if (bad) {
        if (threadIdx.x == 0) atomicExch(&g_tc_error, 1);
    } else if (warp < 16) {
        // flush the weight-gradient accumulators: TMEM lane = this thread's row
        const int row = threadIdx.x & 127, wg = warp >> 2;
        const uint32_t lanef = (uint32_t)(32 * (warp & 3)) << 16;
        float v[16];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            tmem_ld16(tb + kTW3 + lanef + 32 * wg + 16 * k, v);
            if (row < a.ncb)
                red_row<16>(a.dW3 + (size_t)row * kH2 + 32 * wg + 16 * k, v, a.invP, red_vec(a.dW3));
        }
        tmem_ld16(tb + kTW2 + lanef + 16 * wg, v);
        red_row<16>(a.dW2 + (size_t)row * kH1 + 16 * wg, v, a.invP, red_vec(a.dW2));
        if (wg == 0) {
            tmem_ld16(tb + kTP + lanef, v);
            atomicAdd(a.db2 + row, v[0] * a.invP);
            if (row < a.ncb) atomicAdd(a.db3 + row, v[8] * a.invP);
        } else if (wg == 1) {
            tmem_ld16(tb + kTQ + lanef, v);
            if (row < kH1) {
                red_row<kD>(a.dW1 + (size_t)row * kD, v, a.invP, red_vec(a.dW1));
                atomicAdd(a.db1 + row, v[kD] * a.invP);
            }
        }
    }
    if (warp < 16) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            acc_ce += __shfl_xor_sync(0xffffffffu, acc_ce, o);
            acc_u += __shfl_xor_sync(0xffffffffu, acc_u, o);
            acc_l1 += __shfl_xor_sync(0xffffffffu, acc_l1, o);
        }
        if (lane == 0 && ((warp >> 2) & 1) == 0) {
            atomicAdd(a.loss, acc_ce * a.invP);
            atomicAdd(a.loss + 1, acc_u * a.invP);
        }
        if (lane == 0 && ((warp >> 2) & 1) == 1 && a.loss_l1) atomicAdd(a.loss_l1, acc_l1 * a.inv_l1);
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(tb, 512);
}

// ---------------------------------------------------------------------------
// Query (relevancy) and language feature map export, both a decode followed by a
// contraction of the tile's softmax numerators e = exp(z - max z), in BF16, with
// a constant operand B:
//   export  F = M_infer S (supp. Sec. "Inference"): B = the codebook S, each
//           output row scaled by 1 / sum e, BF16 out;
//   query   B = [ [text; negs] S_c^T | S_c S_c^T ]: the projections e.(S_c q) and
//           e^T G, from which |phi|^2 = e^T G e (relevancy does not depend on
//           the scale of e, so its sum is never needed).
// Two 128-pixel tiles are in flight per CTA, each with its own two warpgroups,
// MMA warp and load warp, going through two phases:
//   front  the warpgroups decode the tile and write e over its logits in tensor
//          memory, as the A operand of
//   back   e B in 128-column chunks.  B streams through the tile's four 8 KB
//          slots ([32 codes x 128 columns], bulk copies), the MMA warp contracts
//          them into 128 TMEM columns, and the warpgroups drain a finished
//          chunk, 64 columns each: the export through two 64-byte-swizzled
//          staging boxes and TMA tensor stores (128 pixels x 32 dims), the query
//          into its running e^T G e.
// The second tile starts when the first one enters its back phase, so one tile's
// front, bound by the latency of its rounds, runs beside the other's MMAs and
// stores.  e in tensor memory leaves shared memory for the slots; N = 128 because
// an MMA of N = 64 takes three quarters as long.  Export of a 1296 x 840 view at
// 256 codes: 0.679 ms (2.9 TB/s written); two tiles in phase sharing every slot
// 0.812 ms, the same with e in shared memory 0.886 ms, one tile at a time in rounds
// of two 64-dim chunks 1.255 ms.  Per tile, 45,000 cycles: 17,000 in the front,
// 13,000 waiting for the codebook (the latency of four slots), 13,000 of MMAs.
// A query of 2,073,600 pixels against 256 codes takes 0.714 ms, of 72,261 against
// 64 codes 27 us (0.863 ms and 43 us with one tile at a time, four warpgroups on it
// and G partly resident in shared memory, and the operand's preparation as it was).
constexpr int kXSlots = 4, kXCodes = 32, kXDims = 128;
constexpr uint32_t kXSlotBytes = sbuf_bytes(kXCodes, kXDims), kXBox = sbuf_bytes(128, 32);
// A tile's region: X1 and H1, then H2 over them; in the back phase two staging boxes per warpgroup.
constexpr uint32_t kXAct = sbuf_bytes(128, 128);
static_assert(kXAct == 4 * kXBox && kXAct >= sbuf_bytes(128, 16) + sbuf_bytes(128, 64), "export region");
constexpr int kXThreads = 4 * 128 + 4 * 32;
constexpr uint32_t kXAcc = 128;              // TMEM columns of a tile's 256: e in [0, ncb / 2), the accumulator

struct ExportBars {                          // of one tile slot
    uint64_t full[kXSlots], empty[kXSlots];  // codebook slots
    uint64_t acc_full, acc_free;             // a chunk's accumulator
    uint64_t e_ready;                        // the tile's e is in tensor memory
    uint64_t begun;                          // e_ready of the slot's first tile: completes once
    uint64_t front, fin;
};

// The layout starts at a 1024-byte boundary.
__host__ constexpr size_t export_smem(int ncb)
{
    return 1024 + 2 * kXAct + 2 * kXSlots * kXSlotBytes + weights_bytes(ncb) + 4 * 128 * 4 + 256;
}
static_assert(export_smem(256) <= 227 * 1024 && 2 * sizeof(ExportBars) + 4 <= 256, "export shared memory");

template <bool QUERY>
__device__ __forceinline__ void decode_contract(const CUtensorMap* tmap_out, const DecArgs& a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char* const act =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(sm) + 1023) & ~uintptr_t(1023));
    unsigned char* const slots0 = act + 2 * kXAct;
    const int ncb = a.ncb;
    Front f;
    unsigned char* p = load_weights(slots0 + 2 * kXSlots * kXSlotBytes, a, f);
    float* const sums = reinterpret_cast<float*>(p);              // [tile slot][half][128] partial sums of e
    p += 4 * 128 * 4;
    ExportBars* const bars = reinterpret_cast<ExportBars*>(p);    // [tile slot]
    uint32_t* const tslot = reinterpret_cast<uint32_t*>(bars + 2);
    if (threadIdx.x < 2) {
        ExportBars* const b = bars + threadIdx.x;
        for (int i = 0; i < kXSlots; ++i) {
            mbar_init(b->full + i, 1);
            mbar_init(b->empty + i, 1);
        }
        mbar_init(&b->acc_full, 1);
        mbar_init(&b->acc_free, 8);
        mbar_init(&b->e_ready, 1);
        mbar_init(&b->begun, 1);
        mbar_init(&b->front, 1);
        mbar_init(&b->fin, 1);
    }
    const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (warp == 0) tmem_alloc(tslot, 512);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tbase = warp_uniform(*reinterpret_cast<volatile uint32_t*>(tslot));
    const int ntiles = (a.P + 127) / 128;
    const int nch = (a.dd + kXDims - 1) / kXDims, nkb = (ncb + kXCodes - 1) / kXCodes;
    const auto width = [&](int j) { return min(kXDims, a.dd - j * kXDims); };        // 128, or less in the last chunk
    const auto codes = [&](int k) { return min(kXCodes, ncb - k * kXCodes); };       // 32, or 16 in the last block
    // tile slot t takes the tiles blockIdx.x + gridDim.x (t + 2 i)
    const int t = warp < 16 ? warp >> 3 : warp & 1;
    const int first = blockIdx.x + gridDim.x * t, stride = 2 * gridDim.x;
    ExportBars* const bar = bars + t;
    unsigned char* const slots = slots0 + t * kXSlots * kXSlotBytes;
    const uint32_t td = tbase + 256u * t;
    bool ok = true;

    if (warp >= 18) {
        // B, chunk by chunk, for every tile of the slot
        uint32_t it = 0;
        for (int tile = first; tile < ntiles && ok; tile += stride)
            for (int j = 0; j < nch && ok; ++j) {
                const uint32_t row = (uint32_t)width(j) * 2;
                const unsigned char* src = a.G_img + (size_t)j * ncb * kXDims * 2;
                for (int k = 0; k < nkb; ++k, ++it) {
                    const uint32_t sl = it % kXSlots;
                    if (it >= kXSlots &&
                        !(ok = warp_agree(mbar_wait(bar->empty + sl, (it / kXSlots - 1) & 1u))))
                        break;
                    if (elect_one()) {
                        mbar_expect_tx(bar->full + sl, codes(k) * row);
                        bulk_g2s(slots + sl * kXSlotBytes, src + (size_t)k * kXCodes * row, codes(k) * row,
                                 bar->full + sl);
                    }
                    __syncwarp();
                }
            }
        // copies still in flight land before the shared memory goes away
        for (uint32_t i = it - min(it, (uint32_t)kXSlots); i < it; ++i)
            ok = mbar_wait(bar->full + i % kXSlots, (i / kXSlots) & 1u) && ok;
    } else if (warp >= 16) {
        // the back phase's MMAs
        uint32_t it = 0, r = 0, c = 0;
        const uint32_t slots_a = smem_u32(slots);
        for (int tile = first; tile < ntiles && ok; tile += stride, ++r) {
            if (!(ok = warp_agree(mbar_wait(&bar->e_ready, r & 1u)))) break;
            for (int j = 0; j < nch && ok; ++j, ++c) {
                const uint32_t C = (uint32_t)width(j), id = idesc_bf16((int)C, false, !QUERY);
                if (c >= 1 && !(ok = warp_agree(mbar_wait(&bar->acc_free, (c - 1) & 1u)))) break;
                fence_after();
                for (int k = 0; k < nkb; ++k, ++it) {
                    const uint32_t sl = it % kXSlots;
                    if (!(ok = warp_agree(mbar_wait(bar->full + sl, (it / kXSlots) & 1u)))) break;
                    fence_after();
                    // export: rows are codes (K), read MN-major; query: rows are columns of B (N)
                    const uint32_t at = slots_a + sl * kXSlotBytes;
                    const uint64_t gm = QUERY ? kdesc_at(at, kXCodes, 0, 0) : mndesc_at(at, (int)C, 0, 0);
                    const uint32_t ea = td + 8u * (kXCodes / 16) * k;
                    const bool two = codes(k) > 16;
                    if (elect_one()) {
                        mma_ta(td + kXAcc, ea, gm, id, k > 0);
                        if (two) mma_ta(td + kXAcc, ea + 8u, gm + (QUERY ? 16ull : 2ull * C), id, 1u);
                        commit(bar->empty + sl);
                        if (k + 1 == nkb) commit(&bar->acc_full);
                    }
                    __syncwarp();
                }
            }
        }
        if (elect_one()) commit(&bar->fin);
        ok = mbar_wait(&bar->fin, 0) && ok;
    } else {
        // half h of the tile's columns
        const int wg = warp >> 2;
        f.half = wg & 1;
        f.nhalf = 2;
        f.issuer = (warp & 7) == 0;
        f.tid = threadIdx.x & 127;
        f.bar_id = 1 + t;
        f.nthreads = 256;
        f.mbar = &bar->front;
        f.phase = 0;
        f.tw = td;
        f.lane = (uint32_t)(32 * (warp & 3)) << 16;
        unsigned char* const reg = act + t * kXAct;
        f.X1 = SBuf{reg, 16};
        f.H1 = SBuf{reg + sbuf_bytes(128, 16), 64};
        f.H2 = SBuf{reg, 128};
        f.xch = reinterpret_cast<float4*>(reg);
        const uint32_t tl = f.tw + f.lane;
        unsigned char* const stg = act + wg * 2 * kXBox;
        const int row = f.tid;
        const bool lead = row == 0;                 // of the warpgroup
        // e takes half the logits' columns (two codes a word), so writing it in place must not pass unread
        // logits: each half keeps up to four 16-code units in registers (half 0 its upper ones, whose columns
        // half 1's e will take; half 1 its first ones) until the other has read that far, then goes on in place
        const int nu = ncb / 16, nu0 = (nu + 1) / 2;
        const int u0 = f.half ? nu0 : 0, u1 = f.half ? nu : nu0;
        const int held = f.half ? min(4, nu - nu0) : nu0 - nu0 / 2, hu = f.half ? nu0 : nu0 / 2;
        const int rest0 = f.half ? hu + held : 0, rest1 = f.half ? nu : hu;
        float xf[8];                                // this tile's R_s (half 0), in L2 a tile ahead
        if (f.half == 0) load_feat(a, first * 128 + row, first < ntiles && first * 128 + row < a.P, xf);
        // out of phase with the first slot (a barrier of its own: e_ready's parity comes round again with every
        // second tile, so a thread that looked late would wait for a tile that may not come)
        if (t == 1 && first < ntiles) ok = !bar_any(f.bar_id, 256, !mbar_wait(&bars->begun, 0));
        uint32_t c = 0;
        for (int tile = first; tile < ntiles && ok; tile += stride) {
            const bool valid = tile * 128 + row < a.P;
            if (!(ok = mlp_forward_x(f, a, xf))) break;
            const int nx = tile + stride < ntiles ? (tile + stride) * 128 + row : a.P;
            const bool more = f.half == 0 && nx < a.P;
            if (more)
#pragma unroll
                for (int i = 0; i < 8; ++i) prefetch_l2(a.feat + (size_t)i * a.P + nx);
            float v[16], mh = -INFINITY;
            for (int u = u0; u < u1; ++u) {
                tmem_ld16(tl + 16 * u, v);
                add_bias16(v, f.b3s + 16 * u);
#pragma unroll
                for (int j = 0; j < 16; ++j) mh = fmaxf(mh, v[j]);
            }
            f.xch[f.half * 128 + row].x = mh;
            wg_sync(f);
            const float m = fmaxf(f.xch[row].x, f.xch[128 + row].x);
            const float ml = m * 1.4426950408889634f;
            float se = 0.f;
            const auto unit = [&](int u, uint32_t* w) {
                tmem_ld16(tl + 16 * u, v);
                add_bias16(v, f.b3s + 16 * u);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    v[j] = ex2_approx(fmaf(v[j], 1.4426950408889634f, -ml));
                    se += v[j];
                }
                pack16(v, w);
            };
            uint32_t hold[4][8], w[8];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < held) unit(hu + i, hold[i]);
            fence_before();
            wg_sync(f);
            fence_after();
            if (f.half) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < held) tmem_st8(tl + 8 * (hu + i), hold[i]);
            }
            for (int u = rest0; u < rest1; ++u) {
                unit(u, w);
                tmem_st8(tl + 8 * u, w);
            }
            if (!f.half) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < held) tmem_st8(tl + 8 * (hu + i), hold[i]);
            }
            tmem_wait_st();
            if (!QUERY) sums[wg * 128 + row] = se;
            fence_before();
            wg_sync(f);
            fence_after();
            if (lead && f.half == 0) {
                mbar_arrive(&bar->e_ready);
                if (tile == first) mbar_arrive(&bar->begun);
            }
            const float inv = !QUERY && valid ? 1.0f / (sums[2 * t * 128 + row] + sums[(2 * t + 1) * 128 + row]) : 0.f;
            float pj[16], quad = 0.f;               // query: the projections (half 0), e^T G e over this half's columns
            for (int j = 0; j < nch; ++j, ++c) {
                // the next tile's R_s while the last chunk's MMAs run (the export has no registers to spare here)
                if (QUERY && j + 1 == nch && f.half == 0) load_feat(a, nx, more, xf);
                const bool got = mbar_wait(&bar->acc_full, c & 1u);
                // every thread of the tile leaves together
                if (bar_any(f.bar_id, 256, !got)) {
                    ok = false;
                    break;
                }
                fence_after();
                if constexpr (QUERY) {
                    // 16-column units of the chunk: unit 0 of the first chunk holds the projections, the others
                    // columns of G in order
                    const int w16 = width(j) / 16, wh = (w16 + 1) / 2;
                    for (int u = f.half ? wh : 0; u < (f.half ? w16 : wh); ++u) {
                        tmem_ld16(tl + kXAcc + 16 * u, v);
                        const int col = 8 * j + u - 1;      // unit of G
                        if (col < 0) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) pj[i] = v[i];
                            continue;
                        }
                        tmem_ld8(tl + 8 * col, w);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float2 e2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(w + i));
                            quad = fmaf(e2.x, v[2 * i], quad);
                            quad = fmaf(e2.y, v[2 * i + 1], quad);
                        }
                    }
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar->acc_free);
                } else {
                    const bool mine = 64 * f.half < width(j);
                    __nv_bfloat162 h[32];
                    if (mine) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            tmem_ld16(tl + kXAcc + 64u * f.half + 16u * q, v);
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                h[8 * q + i] = __floats2bfloat162_rn(v[2 * i] * inv, v[2 * i + 1] * inv);
                        }
                    }
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar->acc_free);
                    if (!mine) continue;
                    // row-major 64-byte rows, 16-byte unit u of row r at u ^ ((r >> 1) & 3); a box is rewritten once
                    // the store before the last one has read it
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if (lead) bulk_wait_read_but_one();
                        asm volatile("bar.sync %0, 128;" ::"r"(3 + wg) : "memory");
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            *reinterpret_cast<uint4*>(stg + q * kXBox + row * 64 + ((u ^ ((row >> 1) & 3)) << 4)) =
                                *reinterpret_cast<uint4*>(h + 16 * q + 4 * u);
                        fence_proxy_async();
                        asm volatile("bar.sync %0, 128;" ::"r"(3 + wg) : "memory");
                        if (lead) {
                            tma_store_2d(tmap_out, kXDims * j + 64 * f.half + 32 * q, tile * 128, stg + q * kXBox);
                            bulk_commit();
                        }
                    }
                }
            }
            if (!ok) break;
            if constexpr (QUERY) {
                // the halves' sums meet in shared memory; phi.q / |phi| from the projections
                if (f.half) sums[wg * 128 + row] = quad;
                fence_before();
                wg_sync(f);
                fence_after();
                if (!f.half) {
                    const float inv = rsqrtf(fmaxf(quad + sums[(wg + 1) * 128 + row], 1e-30f));
                    float smax = -INFINITY;
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (i >= a.Q && i < a.Q + a.n_neg) smax = fmaxf(smax, pj[i] * inv);
                    if (valid)
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (i < a.Q)
                                a.rel[(size_t)i * a.P + tile * 128 + row] = 1.f / (1.f + __expf(smax - pj[i] * inv));
                }
                continue;
            }
            if (f.half == 0) load_feat(a, nx, more, xf);
            // the next tile's X1 and H1 go where the staging boxes are
            if (lead) bulk_wait_read_all();
            wg_sync(f);
        }
        if (!QUERY && lead) bulk_wait_all();
    }
    fence_before();
    const bool bad = __syncthreads_or(!ok);
    fence_after();
    if (bad && threadIdx.x == 0) atomicExch(&g_tc_error, 1);
    if (warp == 0) tmem_dealloc(tbase, 512);
}

__global__ void __launch_bounds__(kXThreads, 1) export_fused_kernel(const __grid_constant__ CUtensorMap tmap_out,
                                                                    DecArgs a)
{
    decode_contract<false>(&tmap_out, a);
}

__global__ void __launch_bounds__(kXThreads, 1) query_fused_kernel(DecArgs a) { decode_contract<true>(nullptr, a); }

// The export's codebook S [ncb x dd] (fp32) as a chunked canonical BF16 image:
// chunk j holds dims [128 j, 128 j + 128) (64 in the last chunk of an odd multiple
// of 64) of every code, as an [ncb x 128] canonical buffer, whose blocks of 32
// codes are contiguous.
__global__ void codebook_chunks_kernel(const float* __restrict__ S, int ncb, int dd, unsigned char* __restrict__ img)
{
    const int n8 = ncb * (dd / 8);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += gridDim.x * blockDim.x) {
        const int r = i / (dd / 8), c0 = (i % (dd / 8)) * 8, j = c0 / kXDims;
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = S[(size_t)r * dd + c0 + k];
        const SBuf dst{img + (size_t)j * ncb * kXDims * 2, min(kXDims, dd - j * kXDims)};
        sbuf_store8(dst, r, c0 - j * kXDims, v);
    }
}

// The query's operand B in one launch, 16 x 16 entries per block, k ascending with
// FMAs (the order of a plain dot product), as a chunked BF16 image: chunk j holds
// rows [128 j, 128 j + 128) of
//   rows 0 - 15:     [text; negs] S_c^T (rows past Q + n_neg zero)
//   rows 16 - ...:   G = S_c S_c^T
// in blocks of 32 codes, each an [rows x 32] canonical buffer.  Bound by the latency
// of its loads: 128 columns of both operands a step, read as 16-byte words, the next
// step's loads under this step's products (256 codes against 2,073,600 pixels 730 ->
// 714 us, 64 codes against 72,261 37.2 -> 27.0 us; 32 columns a step, loaded as they
// were needed, and single words before).
__global__ void __launch_bounds__(256) query_prep_kernel(const float* __restrict__ S, int ncb, int dd, int d_clip,
                                                         const float* __restrict__ text, int Q,
                                                         const float* __restrict__ negs, int n_neg,
                                                         unsigned char* __restrict__ img)
{
    constexpr int kK = 128;
    __shared__ __align__(16) float xs[16][kK + 4], ys[16][kK + 4];
    const int j0 = blockIdx.x * 16, i0 = ((int)blockIdx.y - 1) * 16;
    const bool gram = i0 >= 0;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    constexpr int kN = 16 * kK / 256;                // words of each operand per thread and step
    float acc = 0.f, xr[kN], yr[kN];
    const auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < kN; ++q) {
            const int l = threadIdx.x + 256 * q, r = l / kK, k = k0 + l % kK;
            xr[q] = yr[q] = 0.f;
            if (k < d_clip) {
                if (gram) xr[q] = S[(size_t)(i0 + r) * dd + k];
                else if (r < Q) xr[q] = text[(size_t)r * d_clip + k];
                else if (r < Q + n_neg) xr[q] = negs[(size_t)(r - Q) * d_clip + k];
                yr[q] = S[(size_t)(j0 + r) * dd + k];
            }
        }
    };
    load(0);
    for (int k0 = 0; k0 < d_clip; k0 += kK) {
#pragma unroll
        for (int q = 0; q < kN; ++q) {
            const int l = threadIdx.x + 256 * q;
            xs[l / kK][l % kK] = xr[q];
            ys[l / kK][l % kK] = yr[q];
        }
        load(k0 + kK);                               // past the end: zeros, no access
        __syncthreads();
#pragma unroll 8
        for (int c = 0; c < kK; c += 4) {
            const float4 x = *reinterpret_cast<const float4*>(&xs[ty][c]), y = *reinterpret_cast<const float4*>(&ys[tx][c]);
            acc = fmaf(x.x, y.x, acc);
            acc = fmaf(x.y, y.y, acc);
            acc = fmaf(x.z, y.z, acc);
            acc = fmaf(x.w, y.w, acc);
        }
        __syncthreads();
    }
    const int r = i0 + 16 + ty, c = j0 + tx, j = r / kXDims, rows = min(kXDims, 16 + ncb - j * kXDims);
    unsigned char* blk = img + (size_t)j * kXDims * ncb * 2 + (size_t)(c / kXCodes) * rows * kXCodes * 2;
    *reinterpret_cast<__nv_bfloat16*>(blk + sbuf_off(r - j * kXDims, c % kXCodes, kXCodes)) = __float2bfloat16_rn(acc);
}

// Self-test of the bounded-wait path: one thread, not the one that records,
// waits on an mbarrier that nothing ever arrives at, gives up after the usual
// limit, and the block puts the timeout on record.
__global__ void selftest_wait_kernel()
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();
    (void)cta_failed(threadIdx.x != 5 || mbar_wait(&bar, 0u), &g_tc_error);
}

// SM count of the calling thread's current device, read on every launch (a
// cheap attribute query), so a process driving parts of different sizes gets
// each one's own persistent grid.
int sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
        n = 1;
    return n;
}

template <class K>
le_status set_smem(K kernel, size_t bytes)
{
    LE_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return LE_OK;
}

}  // namespace

le_status check_fused_decoder(const le_decoder* d, bool train)
{
    if (d->d_in != kD || d->h1 != kH1 || d->h2 != kH2 || d->n_cb % 16 != 0 || d->n_cb < 16 || d->n_cb > 256 ||
        (train && d->n_cb > 128)) {
        set_error("fused path supports d_in=8, h1=64, h2=128, n_cb multiple of 16 in [16, %d]; got %d-%d-%d-%d",
                  train ? 128 : 256, d->d_in, d->h1, d->h2, d->n_cb);
        return LE_ERR_UNSUPPORTED;
    }
    return LE_OK;
}

size_t decode_fused_workspace(int32_t, const le_decoder*) { return 0; }

le_status decode_fused(int32_t P, const float* feat, const float* unc, const le_decoder* d, const int32_t* target,
                       float lambda_ce, float lambda_u, float* loss, float* d_feat, float* d_unc,
                       const le_decoder_grads* dg, int32_t* argmax, float* prob, void*, size_t, cudaStream_t s,
                       const float* img, const float* img_t, float* loss_l1, float* d_img)
{
    DecArgs a{};
    a.img = img;
    a.img_t = img_t;
    a.loss_l1 = loss_l1;
    a.d_img = d_img;
    a.inv_l1 = 1.0f / (float)(3 * (int64_t)P);
    a.P = P;
    a.ncb = d->n_cb;
    a.feat = feat;
    a.unc = unc;
    a.target = target;
    a.W1 = d->W1; a.b1 = d->b1; a.W2 = d->W2; a.b2 = d->b2; a.W3 = d->W3; a.b3 = d->b3;
    a.lambda_ce = lambda_ce;
    a.lambda_u = lambda_u;
    a.invP = 1.0f / (float)P;
    a.argmax = argmax;
    a.prob = prob;
    const int ntiles = (P + 127) / 128;
    if (target) {
        a.loss = loss; a.d_feat = d_feat; a.d_unc = d_unc;
        a.dW1 = dg->W1; a.db1 = dg->b1; a.dW2 = dg->W2; a.db2 = dg->b2; a.dW3 = dg->W3; a.db3 = dg->b3;
        // the loss and the weight gradients the kernel adds into, zeroed by one launch
        const ZeroList zl{{loss, dg->W1, dg->b1, dg->W2, dg->b2, dg->W3, dg->b3, loss_l1},
                          {2, kH1 * kD, kH1, kH2 * kH1, kH2, a.ncb * kH2, a.ncb, 1}};
        le_status st = zero_list(zl, img ? 8 : 7, s);
        if (st != LE_OK) return st;
        const size_t smem = train_smem(a.ncb);
        if ((st = set_smem(dec_train_kernel, smem)) != LE_OK) return st;
        const int grid = ntiles < sm_count() ? ntiles : sm_count();
        dec_train_kernel<<<grid, kTrainThreads, smem, s>>>(a);
        LE_LAUNCHED();
        return LE_OK;
    }
    const int nwg = a.ncb <= 128 ? 4 : 2, sms = sm_count();
    const size_t smem = fwd_smem(a.ncb, nwg);
    le_status st = nwg == 4 ? set_smem(dec_fwd_kernel<4>, smem) : set_smem(dec_fwd_kernel<2>, smem);
    if (st != LE_OK) return st;
    const int grid = ntiles < sms ? ntiles : sms;
    if (nwg == 4) dec_fwd_kernel<4><<<grid, 512, smem, s>>>(a);
    else dec_fwd_kernel<2><<<grid, 256, smem, s>>>(a);
    LE_LAUNCHED();
    return LE_OK;
}

// The image of the query's operand takes 2 (n_cb + 16) n_cb bytes of this.
size_t query_fused_workspace(int32_t, int32_t n_cb, int32_t)
{
    return align_up(256ull * n_cb, 256) + align_up(sizeof(float) * 16 * n_cb, 256) + align_up(2ull * n_cb * n_cb, 256);
}

le_status query_fused(int32_t P, const float* feat, const le_decoder* d, const float* codebook, int32_t dd,
                      int32_t d_clip, const float* text, int32_t Q, const float* negs, int32_t n_neg, float* rel,
                      void* ws, size_t, cudaStream_t s)
{
    le_status st = check_fused_decoder(d, false);
    if (st != LE_OK) return st;
    const int ncb = d->n_cb;
    if (ncb % 64 != 0) {
        set_error("fused query needs n_cb to be a multiple of 64 (got %d)", ncb);
        return LE_ERR_UNSUPPORTED;
    }
    unsigned char* img = static_cast<unsigned char*>(ws);
    query_prep_kernel<<<dim3(ncb / 16, ncb / 16 + 1), 256, 0, s>>>(codebook, ncb, dd, d_clip, text, Q, negs, n_neg,
                                                                   img);
    LE_LAUNCHED();
    DecArgs a{};
    a.P = P;
    a.ncb = ncb;
    a.feat = feat;
    a.W1 = d->W1; a.b1 = d->b1; a.W2 = d->W2; a.b2 = d->b2; a.W3 = d->W3; a.b3 = d->b3;
    a.G_img = img;
    a.dd = 16 + ncb;
    a.Q = Q;
    a.n_neg = n_neg;
    a.rel = rel;
    const size_t smem = export_smem(ncb);
    if ((st = set_smem(query_fused_kernel, smem)) != LE_OK) return st;
    const int ntiles = (P + 127) / 128, sms = sm_count();
    query_fused_kernel<<<ntiles < sms ? ntiles : sms, kXThreads, smem, s>>>(a);
    LE_LAUNCHED();
    return LE_OK;
}

le_status export_fused(int32_t P, const float* feat, const le_decoder* d, const float* codebook, int32_t dd,
                       __nv_bfloat16* out, void* ws, cudaStream_t s)
{
    le_status st = check_fused_decoder(d, false);
    if (st != LE_OK) return st;
    const int ncb = d->n_cb;
    unsigned char* img = static_cast<unsigned char*>(ws);
    // output tensor map: [P rows, dd columns] BF16, boxes of 128 rows x 32 columns, 64-byte swizzle
    EncodeTiled enc;
    if ((st = tensor_map_encoder(&enc)) != LE_OK) return st;
    CUtensorMap tmap;
    const cuuint64_t dims[2] = {(cuuint64_t)dd, (cuuint64_t)P};
    const cuuint64_t strides[1] = {(cuuint64_t)dd * 2};
    const cuuint32_t box[2] = {32, 128};
    const cuuint32_t estr[2] = {1, 1};
    if (enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, out, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
        CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed for the feature map");
        return LE_ERR_CUDA;
    }
    codebook_chunks_kernel<<<64, 256, 0, s>>>(codebook, ncb, dd, img);
    LE_LAUNCHED();
    DecArgs a{};
    a.P = P;
    a.ncb = ncb;
    a.feat = feat;
    a.W1 = d->W1; a.b1 = d->b1; a.W2 = d->W2; a.b2 = d->b2; a.W3 = d->W3; a.b3 = d->b3;
    a.G_img = img;
    a.dd = dd;
    const size_t smem = export_smem(ncb);
    if ((st = set_smem(export_fused_kernel, smem)) != LE_OK) return st;
    const int ntiles = (P + 127) / 128, sms = sm_count();
    export_fused_kernel<<<ntiles < sms ? ntiles : sms, kXThreads, smem, s>>>(tmap, a);
    LE_LAUNCHED();
    return LE_OK;
}

}  // namespace leg

extern "C" le_status le_feature_map_workspace(int32_t n_cb, int32_t d, size_t* bytes)
{
    LE_TRACE("le_feature_map_workspace");
    LE_CHECK_ARG(bytes != nullptr, "bytes is null");
    LE_CHECK_ARG(n_cb > 0 && d > 0, "bad sizes");
    *bytes = (size_t)n_cb * d * 2 + (size_t)n_cb * 128 * 2;   // the codebook's image; 256 bytes per code to spare
    return LE_OK;
}

extern "C" le_status le_feature_map(int32_t P, const float* feat, const le_decoder* dec, const float* codebook,
                                    int32_t d, uint16_t* out, void* workspace, size_t workspace_bytes, void* stream)
{
    LE_TRACE("le_feature_map");
    LE_CHECK_ARG(P >= 0, "P = %d < 0", P);
    LE_CHECK_ARG(dec != nullptr && codebook && workspace && (P == 0 || out), "null pointer");
    LE_CHECK_ARG(P == 0 || feat != nullptr, "null feat");
    LE_CHECK_ARG(leg::aligned16(out) && leg::aligned16(workspace), "out and workspace must be 16-byte aligned");
    if (d <= 0 || d % 64 != 0) {
        leg::set_error("feature map export needs d to be a positive multiple of 64 (got %d)", d);
        return LE_ERR_UNSUPPORTED;
    }
    LE_CHECK_ARG(workspace_bytes >= (size_t)dec->n_cb * d * 2 + (size_t)dec->n_cb * 128 * 2, "workspace too small");
    if (P == 0) return LE_OK;
    return leg::export_fused(P, feat, dec, codebook, d, reinterpret_cast<__nv_bfloat16*>(out), workspace,
                             leg::as_stream(stream));
}

extern "C" le_status le_selftest_bounded_wait(void* stream)
{
    LE_TRACE("le_selftest_bounded_wait");
    leg::selftest_wait_kernel<<<1, 32, 0, leg::as_stream(stream)>>>();
    LE_LAUNCHED();
    return LE_OK;
}

namespace leg {
le_status quant_take_timeout(bool* timed_out);
le_status smooth_take_timeout(bool* timed_out);
le_status wide_take_timeout(bool* timed_out);
}

extern "C" le_status le_device_status(void* stream)
{
    LE_TRACE("le_device_status");
    LE_CUDA(cudaStreamSynchronize(leg::as_stream(stream)));
    int flag = 0;
    LE_CUDA(cudaMemcpyFromSymbol(&flag, leg::g_tc_error, sizeof(int)));
    bool quant_flag = false;
    const le_status qs = leg::quant_take_timeout(&quant_flag);
    if (qs != LE_OK) return qs;
    bool smooth_flag = false;
    const le_status ss = leg::smooth_take_timeout(&smooth_flag);
    if (ss != LE_OK) return ss;
    bool wide_flag = false;
    const le_status ws = leg::wide_take_timeout(&wide_flag);
    if (ws != LE_OK) return ws;
    if ((quant_flag || smooth_flag || wide_flag) && !flag) {
        leg::set_error(quant_flag    ? "the quantisation kernel gave up on a bounded wait"
                       : smooth_flag ? "the smoothing kernel gave up on a bounded wait"
                                     : "a decoder kernel at the widths 8-128-256-N gave up on a bounded wait");
        return LE_ERR_TIMEOUT;
    }
    if (flag) {
        const int zero = 0;
        LE_CUDA(cudaMemcpyToSymbol(leg::g_tc_error, &zero, sizeof(int)));
        leg::set_error("a tensor-core kernel gave up on a bounded wait");
        return LE_ERR_TIMEOUT;
    }
    return LE_OK;
}
