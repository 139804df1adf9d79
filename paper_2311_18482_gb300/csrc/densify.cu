// Adaptive density control of 3D Gaussian Splatting, which Sec. 4 keeps
// (clone / split / prune, opacity reset), as the steps the training loop calls:
//   le_densify_stats  every step: acc_i += |dL/dmean2d_i| (pixels), cnt_i += 1
//                     and max_radius_i = max(max_radius_i, radius_i) for every
//                     Gaussian with a nonzero screen radius;
//   le_opacity_reset  every few thousand steps: opacity = min(opacity, 0.01),
//                     the opacity's Adam moments zeroed;
//   le_densify        every few hundred steps: classify each Gaussian (pruned,
//                     kept, kept + clone, split), count the three output
//                     segments per block, scan the block counts, then scatter
//                     parameters and Adam moments into the caller's output
//                     arrays: kept and cloned Gaussians (index order), clones
//                     (index order), two children per split Gaussian.
// The decisions use FP32 comparisons against thresholds derived once in double
// (no transcendental function on the device), so they are reproducible bit for
// bit: opacity_raw < logit(min_opacity); max log-scale > ln(percent_dense *
// extent); cnt > 0 and acc >= fl(grad_thresh * cnt); and, when enabled, the
// size tests that prune Gaussians too large on screen (max_radius >
// max_screen_size) or in the world (max log-scale > ln(world_frac * extent)).  A split child k copies
// its parent except mean = mu + R(q) diag(exp(log-scale)) n_k (the caller's
// standard normal samples) and log-scale - ln(1.6); clones and children start
// with zero Adam moments.
#include "common.cuh"

namespace leg {
namespace {

constexpr int kDB = 1024;                  // Gaussians per classification block
constexpr int kSB = 512;                   // Gaussians per scatter block

struct DensifyThresholds {
    float grad_thresh, log_big, logit_min, ln16, max_screen, log_world;
};

struct Fields {
    float* f[7];
};

__global__ void densify_stats_kernel(int n, const float4* __restrict__ grad2d, const int* __restrict__ radius,
                                     float* __restrict__ acc, int* __restrict__ cnt, int* __restrict__ max_radius)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int r = radius[i];
    if (r <= 0) return;
    const float4 g = grad2d[5 * (size_t)i];
    acc[i] = __fadd_rn(acc[i], __fsqrt_rn(__fadd_rn(__fmul_rn(g.x, g.x), __fmul_rn(g.y, g.y))));
    cnt[i] += 1;
    if (max_radius && r > max_radius[i]) max_radius[i] = r;
}

// opacity_raw = min(opacity_raw, logit_max); the opacity's Adam moments zeroed.
__global__ void opacity_reset_kernel(int n, float* __restrict__ op, float* __restrict__ m, float* __restrict__ v,
                                     float logit_max)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    op[i] = fminf(op[i], logit_max);
    m[i] = 0.f;
    v[i] = 0.f;
}

__device__ __forceinline__ int classify(int i, const float* ls, const float* op, const float* acc, const int* cnt,
                                        const int* max_radius, const DensifyThresholds& t)
{
    const float smax = fmaxf(fmaxf(ls[3 * i], ls[3 * i + 1]), ls[3 * i + 2]);
    const int c = cnt[i];
    const bool cand = c > 0 && acc[i] >= __fmul_rn(t.grad_thresh, (float)c);
    const bool big_screen = t.max_screen > 0.f && (float)max_radius[i] > t.max_screen;
    if (op[i] < t.logit_min || big_screen || smax > t.log_world) return 0;
    if (cand) return smax > t.log_big ? 3 : 2;
    return 1;
}

// kind[i] and per-block counts of the three output segments: [3][nblocks].
__global__ void __launch_bounds__(256) densify_count_kernel(int n, const float* __restrict__ ls,
                                                            const float* __restrict__ op, const float* __restrict__ acc,
                                                            const int* __restrict__ cnt,
                                                            const int* __restrict__ max_radius, DensifyThresholds t,
                                                            uint8_t* __restrict__ kind, unsigned* __restrict__ bcount)
{
    __shared__ unsigned c3[3];
    if (threadIdx.x < 3) c3[threadIdx.x] = 0;
    __syncthreads();
    unsigned k1 = 0, k2 = 0, k3 = 0;
    for (int r = 0; r < kDB / 256; ++r) {
        const int i = blockIdx.x * kDB + r * 256 + threadIdx.x;
        if (i < n) {
            const int k = classify(i, ls, op, acc, cnt, max_radius, t);
            kind[i] = (uint8_t)k;
            k1 += k == 1 || k == 2;
            k2 += k == 2;
            k3 += k == 3;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        k1 += __shfl_xor_sync(0xffffffffu, k1, o);
        k2 += __shfl_xor_sync(0xffffffffu, k2, o);
        k3 += __shfl_xor_sync(0xffffffffu, k3, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&c3[0], k1);
        atomicAdd(&c3[1], k2);
        atomicAdd(&c3[2], k3);
    }
    __syncthreads();
    if (threadIdx.x < 3) bcount[threadIdx.x * gridDim.x + blockIdx.x] = c3[threadIdx.x];
}

// Exclusive scan of each segment's block counts, in place; totals[3].  One block.
__global__ void __launch_bounds__(1024) densify_scan_kernel(unsigned* bcount, int nb, unsigned long long* totals)
{
    __shared__ unsigned long long carry;
    __shared__ unsigned wsum[32];
    for (int sgm = 0; sgm < 3; ++sgm) {
        unsigned* c = bcount + (size_t)sgm * nb;
        if (threadIdx.x == 0) carry = 0;
        __syncthreads();
        for (int b0 = 0; b0 < nb; b0 += 1024) {
            const int b = b0 + threadIdx.x;
            const unsigned v = b < nb ? c[b] : 0u;
            unsigned x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
                if ((threadIdx.x & 31) >= o) x += y;
            }
            if ((threadIdx.x & 31) == 31) wsum[threadIdx.x >> 5] = x;
            __syncthreads();
            if (threadIdx.x < 32) {
                unsigned w = wsum[threadIdx.x];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, w, o);
                    if (threadIdx.x >= o) w += y;
                }
                wsum[threadIdx.x] = w;
            }
            __syncthreads();
            const unsigned incl = x + ((threadIdx.x >> 5) > 0 ? wsum[(threadIdx.x >> 5) - 1] : 0u);
            if (b < nb) c[b] = (unsigned)(carry + incl - v);
            __syncthreads();
            if (threadIdx.x == 1023) carry += incl;
            __syncthreads();
        }
        if (threadIdx.x == 0) totals[sgm] = carry;
        __syncthreads();
    }
}

struct ScatterArgs {
    int n, nb;                      // Gaussians, classification blocks
    Fields p, m, v;                 // inputs
    Fields po, mo, vo;              // outputs
    const uint8_t* kind;
    const unsigned* boff;           // [3][nblocks] exclusive block offsets
    const unsigned long long* totals;
    const float* noise;             // [n][2][3]
    float ln16;
    unsigned vec;                   // bit f: the six arrays of field f are 16-byte aligned
};

// The block's Gaussians of one output segment: their indices within the block,
// in order, and the segment's first output slot.
struct Segment {
    const uint16_t* list;
    int count;
    size_t dst;
};

constexpr int kCopyUnroll = 4;             // units of a field in flight per thread, times three arrays

// One field of WIDTH units T per Gaussian (float4 for rows of whole 16 bytes,
// else float), for the block's kept Gaussians (parameters and moments) and its
// clones and children (parameters; zero moments).  Output rows are consecutive,
// so unit t of the segment goes to unit t of a contiguous range and the
// accesses of a warp are consecutive 4- or 16-byte units on both sides (reads
// break only where a Gaussian is left out).
template <typename T, int WIDTH>
__device__ __forceinline__ void copy_rows(const ScatterArgs& a, int f, size_t base, const Segment& kept,
                                          const Segment& clone, const Segment& split)
{
    const T* __restrict__ ps = reinterpret_cast<const T*>(a.p.f[f]) + base * WIDTH;
    const T* __restrict__ ms = reinterpret_cast<const T*>(a.m.f[f]) + base * WIDTH;
    const T* __restrict__ vs = reinterpret_cast<const T*>(a.v.f[f]) + base * WIDTH;
    T* __restrict__ pd = reinterpret_cast<T*>(a.po.f[f]);
    T* __restrict__ md = reinterpret_cast<T*>(a.mo.f[f]);
    T* __restrict__ vd = reinterpret_cast<T*>(a.vo.f[f]);
    const int nk = kept.count * WIDTH;
    const size_t dk = kept.dst * WIDTH;
    for (int t0 = threadIdx.x; t0 < nk; t0 += kCopyUnroll * 256) {
        T rp[kCopyUnroll], rm[kCopyUnroll], rv[kCopyUnroll];
#pragma unroll
        for (int u = 0; u < kCopyUnroll; ++u) {
            const int t = t0 + 256 * u;
            if (t < nk) {
                const int o = kept.list[t / WIDTH] * WIDTH + t % WIDTH;
                rp[u] = __ldcs(ps + o);
                rm[u] = __ldcs(ms + o);
                rv[u] = __ldcs(vs + o);
            }
        }
#pragma unroll
        for (int u = 0; u < kCopyUnroll; ++u) {
            const int t = t0 + 256 * u;
            if (t < nk) {
                __stcs(pd + dk + t, rp[u]);
                __stcs(md + dk + t, rm[u]);
                __stcs(vd + dk + t, rv[u]);
            }
        }
    }
    const T zero = T();
    const int nc = clone.count * WIDTH;
    const size_t dc = clone.dst * WIDTH;
    for (int t = threadIdx.x; t < nc; t += 256) {
        pd[dc + t] = ps[clone.list[t / WIDTH] * WIDTH + t % WIDTH];
        __stcs(md + dc + t, zero);
        __stcs(vd + dc + t, zero);
    }
    const int ns = 2 * split.count * WIDTH;
    const size_t ds = split.dst * WIDTH;
    for (int t = threadIdx.x; t < ns; t += 256) {
        if (f > 1) pd[ds + t] = ps[split.list[t / (2 * WIDTH)] * WIDTH + t % WIDTH];   // means, scales: child_rows
        __stcs(md + ds + t, zero);
        __stcs(vd + ds + t, zero);
    }
}

// Means and log-scales of the block's split children, one thread per child.
__device__ __forceinline__ void child_rows(const ScatterArgs& a, size_t base, const Segment& split)
{
    for (int t = threadIdx.x; t < 2 * split.count; t += 256) {
        const size_t i = base + split.list[t >> 1];
        const float* q = a.p.f[2] + 4 * i;
        const float* ls = a.p.f[1] + 3 * i;
        const float* mu = a.p.f[0] + 3 * i;
        const float qn = rsqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
        const float w = q[0] * qn, x = q[1] * qn, y = q[2] * qn, z = q[3] * qn;
        const float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y)},
                               {2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x)},
                               {2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)}};
        const float s[3] = {expf(ls[0]), expf(ls[1]), expf(ls[2])};
        const float* nz = a.noise + 6 * i + 3 * (t & 1);
        const float v0 = s[0] * nz[0], v1 = s[1] * nz[1], v2 = s[2] * nz[2];
        float* mo = a.po.f[0] + 3 * (split.dst + t);
        float* lo = a.po.f[1] + 3 * (split.dst + t);
#pragma unroll
        for (int rr = 0; rr < 3; ++rr) {
            mo[rr] = mu[rr] + R[rr][0] * v0 + R[rr][1] * v1 + R[rr][2] * v2;
            lo[rr] = ls[rr] - a.ln16;
        }
    }
}

// Lists the block's Gaussians of each segment (a block-wide scan of the three
// flags, in index order; the block of a classification block's second half
// counts the first half's for its offsets), then copies field by field.  A
// copy bound by HBM: at 1M Gaussians of SH degree 3 (900k left, 1.13M out) it
// reads and writes 1.7 GB.  One thread per Gaussian walking its own rows
// touched 32 rows per warp instruction (the whole call took 0.733 ms); rows
// dealt out by output unit make every warp access consecutive (0.333 ms).  While
// all blocks are resident anyway, each field has blocks of its own.
template <int NC>
__global__ void __launch_bounds__(256) densify_scatter_kernel(ScatterArgs a)
{
    __shared__ unsigned wsum[3][8];
    __shared__ uint16_t list[3][kSB];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cb = blockIdx.x / (kDB / kSB), first = blockIdx.x % (kDB / kSB) * kSB;
    const size_t base = (size_t)blockIdx.x * kSB;
    unsigned run[3] = {0, 0, 0}, skip[3] = {0, 0, 0};
    for (int r = 0; r < (first + kSB) / 256; ++r) {
        const int l = r * 256 + threadIdx.x - first;          // < 0: the classification block's earlier half
        if (r * 256 == first)
            for (int s = 0; s < 3; ++s) {
                skip[s] = run[s];
                run[s] = 0;
            }
        const long long i = (long long)base + l;
        const int k = i < a.n ? a.kind[i] : 0;
        const bool f[3] = {k == 1 || k == 2, k == 2, k == 3};
        unsigned before[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const unsigned b = __ballot_sync(0xffffffffu, f[s]);
            before[s] = __popc(b & ((1u << lane) - 1u));
            if (lane == 0) wsum[s][warp] = __popc(b);
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            unsigned all = 0;
            for (int w = 0; w < 8; ++w) {
                if (w < warp) before[s] += wsum[s][w];
                all += wsum[s][w];
            }
            if (f[s] && l >= 0) list[s][run[s] + before[s]] = (uint16_t)l;
            run[s] += all;
        }
        __syncthreads();
    }
    const size_t K1 = a.totals[0], K2 = a.totals[1];
    const Segment kept = {list[0], (int)run[0], (size_t)(a.boff[cb] + skip[0])};
    const Segment clone = {list[1], (int)run[1], K1 + a.boff[(size_t)a.nb + cb] + skip[1]};
    const Segment split = {list[2], (int)run[2], K1 + K2 + 2 * (size_t)(a.boff[2 * (size_t)a.nb + cb] + skip[2])};
    // a field moves in 16-byte units when its rows are whole multiples of them and its six arrays are aligned
    const auto mine = [](int f) { return gridDim.y == 1 || (int)blockIdx.y == f; };
    if (mine(0)) {
        copy_rows<float, 3>(a, 0, base, kept, clone, split);
        child_rows(a, base, split);
    }
    if (mine(1)) copy_rows<float, 3>(a, 1, base, kept, clone, split);
    if (mine(2)) {
        if (a.vec & 4u) copy_rows<float4, 1>(a, 2, base, kept, clone, split);
        else copy_rows<float, 4>(a, 2, base, kept, clone, split);
    }
    if (mine(3)) copy_rows<float, 1>(a, 3, base, kept, clone, split);
    if (mine(4)) {
        if constexpr (3 * NC % 4 == 0) {
            if (a.vec & 16u) copy_rows<float4, 3 * NC / 4>(a, 4, base, kept, clone, split);
            else copy_rows<float, 3 * NC>(a, 4, base, kept, clone, split);
        } else {
            copy_rows<float, 3 * NC>(a, 4, base, kept, clone, split);
        }
    }
    if (mine(5)) {
        if (a.vec & 32u) copy_rows<float4, 2>(a, 5, base, kept, clone, split);
        else copy_rows<float, 8>(a, 5, base, kept, clone, split);
    }
    if (mine(6)) copy_rows<float, 1>(a, 6, base, kept, clone, split);
}

Fields fields_of(const le_gaussian_grads* g)
{
    Fields f;
    float* const p[7] = {g->means, g->log_scales, g->quats, g->opacity_raw, g->sh, g->feat, g->unc};
    for (int i = 0; i < 7; ++i) f.f[i] = p[i];
    return f;
}

bool fields_ok(const le_gaussian_grads* g)
{
    return g && g->means && g->log_scales && g->quats && g->opacity_raw && g->sh && g->feat && g->unc;
}

}  // namespace
}  // namespace leg

using namespace leg;

extern "C" le_status le_densify_stats(int32_t n, const float* grad2d, const int32_t* radius, float* acc, int32_t* cnt,
                                      int32_t* max_radius, void* stream)
{
    LE_TRACE("le_densify_stats");
    LE_CHECK_ARG(n >= 0, "n = %d < 0", n);
    if (n == 0) return LE_OK;
    LE_CHECK_ARG(grad2d && radius && acc && cnt, "null pointer");
    LE_CHECK_ARG(aligned16(grad2d), "grad2d must be 16-byte aligned");
    densify_stats_kernel<<<(n + 255) / 256, 256, 0, as_stream(stream)>>>(n, reinterpret_cast<const float4*>(grad2d),
                                                                         radius, acc, cnt, max_radius);
    LE_LAUNCHED();
    return LE_OK;
}

extern "C" le_status le_opacity_reset(int32_t n, float* opacity_raw, float* m_opacity, float* v_opacity,
                                      float max_opacity, void* stream)
{
    LE_TRACE("le_opacity_reset");
    LE_CHECK_ARG(n >= 0, "n = %d < 0", n);
    LE_CHECK_ARG(max_opacity > 0.f && max_opacity < 1.f, "max_opacity = %g outside (0, 1)", (double)max_opacity);
    if (n == 0) return LE_OK;
    LE_CHECK_ARG(opacity_raw && m_opacity && v_opacity, "null pointer");
    const float logit_max = (float)log((double)max_opacity / (1.0 - (double)max_opacity));
    opacity_reset_kernel<<<(n + 255) / 256, 256, 0, as_stream(stream)>>>(n, opacity_raw, m_opacity, v_opacity,
                                                                         logit_max);
    LE_LAUNCHED();
    return LE_OK;
}

extern "C" le_status le_densify_workspace(int32_t n, size_t* bytes)
{
    LE_TRACE("le_densify_workspace");
    LE_CHECK_ARG(bytes != nullptr && n >= 0, "bad arguments");
    const size_t nb = ((size_t)n + kDB - 1) / kDB;
    *bytes = ((size_t)n + 255) / 256 * 256 + (3 * nb * 4 + 255) / 256 * 256 + 256;
    return LE_OK;
}

extern "C" le_status le_densify(const le_densify_config* cfg, const le_gaussians* g, const le_gaussian_grads* m,
                                const le_gaussian_grads* v, const float* acc, const int32_t* cnt,
                                const int32_t* max_radius, const float* noise,
                                int64_t n_cap, const le_gaussian_grads* g_out, const le_gaussian_grads* m_out,
                                const le_gaussian_grads* v_out, int64_t* n_out, void* workspace,
                                size_t workspace_bytes, void* stream)
{
    LE_TRACE("le_densify");
    LE_CHECK_ARG(cfg && g && n_out, "null config / gaussians / n_out");
    LE_CHECK_ARG(g->n >= 0 && g->sh_degree >= 0 && g->sh_degree <= 3, "bad gaussians");
    LE_CHECK_ARG(cfg->min_opacity > 0.f && cfg->min_opacity < 1.f && cfg->percent_dense > 0.f &&
                     cfg->scene_extent > 0.f && cfg->grad_thresh >= 0.f && cfg->max_screen_size >= 0.f &&
                     cfg->world_frac >= 0.f,
                 "bad densify config");
    const int n = g->n;
    if (n == 0) {
        *n_out = 0;
        return LE_OK;
    }
    LE_CHECK_ARG(g->means && g->log_scales && g->quats && g->opacity_raw && g->sh && g->feat && g->unc,
                 "null Gaussian parameter");
    LE_CHECK_ARG(fields_ok(m) && fields_ok(v) && fields_ok(g_out) && fields_ok(m_out) && fields_ok(v_out),
                 "null moment / output pointer");
    LE_CHECK_ARG(acc && cnt && noise && workspace, "null statistics / noise / workspace");
    LE_CHECK_ARG(cfg->max_screen_size == 0.f || max_radius, "max_screen_size > 0 needs max_radius");
    size_t need = 0;
    le_densify_workspace(n, &need);
    LE_CHECK_ARG(workspace_bytes >= need, "workspace has %zu bytes, needs %zu", workspace_bytes, need);
    LE_CHECK_ARG((reinterpret_cast<uintptr_t>(workspace) & 7u) == 0, "workspace must be 8-byte aligned");
    const int nb = (n + kDB - 1) / kDB;
    unsigned char* w = static_cast<unsigned char*>(workspace);
    uint8_t* kind = w;
    unsigned* bcount = reinterpret_cast<unsigned*>(w + ((size_t)n + 255) / 256 * 256);
    unsigned long long* totals =
        reinterpret_cast<unsigned long long*>(w + ((size_t)n + 255) / 256 * 256 + (3 * (size_t)nb * 4 + 255) / 256 * 256);
    DensifyThresholds t;
    t.grad_thresh = cfg->grad_thresh;
    t.log_big = (float)log((double)cfg->percent_dense * (double)cfg->scene_extent);
    t.logit_min = (float)log((double)cfg->min_opacity / (1.0 - (double)cfg->min_opacity));
    t.ln16 = (float)log(1.6);
    t.max_screen = cfg->max_screen_size;
    t.log_world = cfg->world_frac > 0.f ? (float)log((double)cfg->world_frac * (double)cfg->scene_extent) : INFINITY;
    cudaStream_t s = as_stream(stream);
    densify_count_kernel<<<nb, 256, 0, s>>>(n, g->log_scales, g->opacity_raw, acc, cnt, max_radius, t, kind,
                                            bcount);
    LE_LAUNCHED();
    densify_scan_kernel<<<1, 1024, 0, s>>>(bcount, nb, totals);
    LE_LAUNCHED();
    unsigned long long h[3];
    LE_CUDA(cudaMemcpyAsync(h, totals, sizeof(h), cudaMemcpyDeviceToHost, s));
    LE_CUDA(cudaStreamSynchronize(s));
    const unsigned long long total = h[0] + h[1] + 2 * h[2];
    *n_out = (int64_t)total;
    if ((long long)total > n_cap) {
        set_error("densify: %llu Gaussians after densification exceed the capacity %lld", total, (long long)n_cap);
        return LE_ERR_CAPACITY;
    }
    ScatterArgs a;
    a.n = n;
    float* const gp[7] = {const_cast<float*>(g->means), const_cast<float*>(g->log_scales), const_cast<float*>(g->quats),
                          const_cast<float*>(g->opacity_raw), const_cast<float*>(g->sh), const_cast<float*>(g->feat),
                          const_cast<float*>(g->unc)};
    for (int i = 0; i < 7; ++i) a.p.f[i] = gp[i];
    a.m = fields_of(m);
    a.v = fields_of(v);
    a.po = fields_of(g_out);
    a.mo = fields_of(m_out);
    a.vo = fields_of(v_out);
    a.kind = kind;
    a.boff = bcount;
    a.totals = totals;
    a.noise = noise;
    a.ln16 = t.ln16;
    a.nb = nb;
    a.vec = 0;
    for (int i = 0; i < 7; ++i)
        if (aligned16(a.p.f[i]) && aligned16(a.m.f[i]) && aligned16(a.v.f[i]) && aligned16(a.po.f[i]) &&
            aligned16(a.mo.f[i]) && aligned16(a.vo.f[i]))
            a.vec |= 1u << i;
    // up to here seven blocks per 512 Gaussians are resident at once (152 SMs x 8 blocks)
    const int blocks = (n + kSB - 1) / kSB;
    const dim3 sb(blocks, 7 * blocks <= 152 * 8 ? 7 : 1);
    switch (g->sh_degree) {
        case 0: densify_scatter_kernel<1><<<sb, 256, 0, s>>>(a); break;
        case 1: densify_scatter_kernel<4><<<sb, 256, 0, s>>>(a); break;
        case 2: densify_scatter_kernel<9><<<sb, 256, 0, s>>>(a); break;
        default: densify_scatter_kernel<16><<<sb, 256, 0, s>>>(a); break;
    }
    LE_LAUNCHED();
    return LE_OK;
}
