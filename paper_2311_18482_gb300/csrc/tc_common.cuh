// tcgen05 / TMEM / mbarrier building blocks (inline PTX, sm_100-family).
//
// Shared-memory operands use the no-swizzle canonical layout: a bf16 matrix
// X[r][c] with C columns is stored as 8x8 core matrices of 8 rows x 16 bytes,
//   off(r, c) = (r/8) * (C/8) * 128 + (c/8) * 128 + (r%8) * 16 + (c%8) * 2.
// Read K-major (rows = M or N, columns = K) its descriptor has LBO = 128 (core
// stride along K) and SBO = (C/8)*128 (stride between 8-row groups); read
// MN-major (rows = K, columns = M or N) LBO = (C/8)*128 (stride along K) and
// SBO = 128.  In both cases LBO is the stride between core matrices adjacent
// in K and SBO the one between core matrices adjacent in M/N.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"

namespace leg {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Named barrier over `n` threads; returns whether any participating thread passed pred = true.
__device__ __forceinline__ bool bar_any(int id, int n, bool pred)
{
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}\n"
                 : "=r"(r)
                 : "r"((uint32_t)pred), "r"(id), "r"(n)
                 : "memory");
    return r != 0;
}

__device__ __forceinline__ void mbar_init(uint64_t* m, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count) : "memory");
}

// Bounded wait for the phase with the given parity to complete.  Gives up
// after ~2^31 SM cycles (about a second) and returns false.  The try_wait
// carries a suspend-time hint, so the waiting thread sleeps in the barrier
// until the phase completes instead of spinning on issue slots.
__device__ __forceinline__ bool mbar_wait(uint64_t* m, uint32_t parity)
{
    const uint32_t a = smem_u32(m);
    const long long t0 = clock64();
    while (true) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity), "r"(0x989680u)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > (1ll << 31)) return false;
    }
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* m, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(m)), "r"(bytes) : "memory");
}

// 1-D bulk copy global -> this CTA's shared memory, completion counted on m.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* m)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(m))
                 : "memory");
}

// 2-D tensor store shared -> global through the tensor map (TMA), counted in
// this thread's bulk async-group; elements outside the tensor are not written.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, const void* src)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(smem_u32(src))
                 : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

// Until all but the last of this thread's committed bulk stores have read their shared-memory source.
__device__ __forceinline__ void bulk_wait_read_but_one() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }

// Until this thread's committed bulk stores have read their shared-memory source.
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// Until this thread's committed bulk stores have completed.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Warp-wide TMEM allocation; the base address is written to *slot.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// kind::f16 instruction descriptor: BF16 A and B, FP32 accumulator, M = 128.
__host__ __device__ constexpr uint32_t idesc_bf16(int N, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ uint64_t make_desc(uint32_t start, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((start & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// MMAs are issued by one lane, but from code that the whole warp runs:
//   if (warp == k) { ...loop, waits, descriptors...; if (elect_one()) { mma(...); commit(...); } }
// with the warp index and the TMEM base made warp-uniform by warp_uniform().
// The descriptors then live in uniform registers, where tcgen05.mma takes them
// from.  Under a lane == 0 branch each one is moved there by its own
// instruction and the loop runs on one lane's vector registers: 125 cycles per
// M = 128, K = 16 MMA whatever N is, against 53 (N = 64) and 66 (N = 128), the
// tensor core's own rate (le_smooth on 1M Gaussians 0.584 -> 0.527 ms; the
// decoder kernels, bound by other parts of a tile, 2 to 3 %).  A warp's MMAs
// and commits all come from the same elected lane.
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
    return r != 0;
}

__device__ __forceinline__ uint32_t warp_uniform(uint32_t x) { return __shfl_sync(0xffffffffu, x, 0); }

// A wait done by a whole warp: one outcome for all lanes, so that a timeout never
// leaves part of them at the next elect_one().
__device__ __forceinline__ bool warp_agree(bool ok) { return __all_sync(0xffffffffu, ok); }

// A barrier of the whole CTA that joins its threads' outcomes: true for all if any of them gave up, which is
// then on record (each thread has a clock of its own, so any one of them may be the only one).
__device__ __forceinline__ bool cta_failed(bool ok, int* error)
{
    const bool bad = __syncthreads_or(!ok);
    if (bad && threadIdx.x == 0) atomicExch(error, 1);
    return bad;
}

// D[tmem] (+)= A * B, issued by one thread.
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                     d_tmem),
                 "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
                 : "memory");
}

// The same with A in tensor memory: row r of A in lane r, two consecutive BF16
// K elements per 32-bit column.
__device__ __forceinline__ void mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(
                     d_tmem),
                 "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate)
                 : "memory");
}

// mbarrier arrives once all tcgen05 operations issued so far by this thread complete.
__device__ __forceinline__ void commit(uint64_t* m)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(m))
                 : "memory");
}

// 16 consecutive FP32 columns of this thread's TMEM lane.  The load and its
// wait are one asm statement, so no use of the registers can be scheduled
// before the data has arrived.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v)
{
    uint32_t r[16];
    asm volatile(
        "{\ntcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n}\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// 8 consecutive words of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r)
{
    asm volatile(
        "{\ntcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
        "tcgen05.wait::ld.sync.aligned;\n}\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr)
        : "memory");
}

// Store 16 FP32 values to consecutive columns of this thread's TMEM lane; call
// tmem_wait_st() before reading them back.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
        "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
        "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])),
        "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])),
        "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
        : "memory");
}

// Store 8 words to consecutive columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Single arrival on an mbarrier (release semantics at CTA scope).
__device__ __forceinline__ void mbar_arrive(uint64_t* m)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(m)) : "memory");
}


// ---------------------------------------------------------------------------
// Canonical no-swizzle bf16 buffer in shared memory.
struct SBuf {
    unsigned char* p;
    int C;   // columns (multiple of 8)
};

__host__ __device__ constexpr uint32_t sbuf_bytes(int R, int C) { return (uint32_t)R * C * 2; }

__device__ __forceinline__ uint32_t sbuf_off(int r, int c, int C)
{
    return (uint32_t)((r >> 3) * (C >> 3) * 128 + (c >> 3) * 128 + (r & 7) * 16 + (c & 7) * 2);
}

// 8 consecutive columns [c0, c0+8) of row r (c0 multiple of 8) in one 16-byte store.
__device__ __forceinline__ void sbuf_store8(const SBuf& b, int r, int c0, const float* v)
{
    __nv_bfloat162 h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    *reinterpret_cast<uint4*>(b.p + sbuf_off(r, c0, b.C)) = *reinterpret_cast<uint4*>(h);
}

// Descriptor of the (128-row or N-row) K-major block whose first row is row0,
// K columns starting at k0 (both multiples of 8).
__device__ __forceinline__ uint64_t kdesc(const SBuf& b, int row0, int k0)
{
    return make_desc(smem_u32(b.p) + sbuf_off(row0, k0, b.C), 128u, (uint32_t)(b.C >> 3) * 128u);
}

// The same for a buffer given by its shared-memory address and column count, and
// the MN-major block: rows are K (starting at k0), columns are M/N (starting at mn0).
__device__ __forceinline__ uint64_t kdesc_at(uint32_t base, int C, int row0, int k0)
{
    return make_desc(base + sbuf_off(row0, k0, C), 128u, (uint32_t)(C >> 3) * 128u);
}

__device__ __forceinline__ uint64_t mndesc_at(uint32_t base, int C, int k0, int mn0)
{
    return make_desc(base + sbuf_off(k0, mn0, C), (uint32_t)(C >> 3) * 128u, 128u);
}

// Epilogue arithmetic on pairs: a layer's epilogue is bound by issue slots, so
// bias comes in 16-byte loads, the ReLU and its mask work on two BF16 values an
// instruction, and a backward epilogue reads the layer's own output again as the
// mask (max(x, 0) rounded to BF16 is positive where x is) instead of keeping a
// bit per value, which cost three instructions forward and two backward (le_smooth
// on 1M Gaussians 0.527 -> 0.490 ms, the training step at 1M 1.450 -> 1.413 ms).

// v += b (b 16-byte aligned).
__device__ __forceinline__ void add_bias16(float* v, const float* b)
{
#pragma unroll
    for (int j = 0; j < 16; j += 4) {
        const float4 w = *reinterpret_cast<const float4*>(b + j);
        v[j] += w.x;
        v[j + 1] += w.y;
        v[j + 2] += w.z;
        v[j + 3] += w.w;
    }
}

// 16 floats as eight BF16 pairs.
__device__ __forceinline__ void pack16(const float* v, uint32_t* w)
{
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        w[j] = *reinterpret_cast<const uint32_t*>(&b);
    }
}

__device__ __forceinline__ uint32_t relu2(uint32_t w)
{
    const __nv_bfloat162 b = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&w), __nv_bfloat162());
    return *reinterpret_cast<const uint32_t*>(&b);
}

// 0xFFFF in the halves of w that are positive.
__device__ __forceinline__ uint32_t positive2(uint32_t w)
{
    return __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&w), __nv_bfloat162());
}

// relu(v + b) as BF16 pairs.
__device__ __forceinline__ void relu16(float* v, const float* b, uint32_t* w)
{
    add_bias16(v, b);
    pack16(v, w);
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = relu2(w[j]);
}

__device__ __forceinline__ void sts128(uint32_t addr, const uint32_t* w)
{
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                 : "memory");
}

__device__ __forceinline__ void lds128(uint32_t addr, uint32_t* w)
{
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                 : "r"(addr)
                 : "memory");
}

// 16 columns of a canonical row whose first 16-byte unit is at addr (the second follows at 128).
__device__ __forceinline__ void sts_row16(uint32_t addr, const uint32_t* w)
{
    sts128(addr, w);
    sts128(addr + 128, w + 4);
}

// Whether red_row may use 16-byte reductions at p (and at every row of whole 16 bytes behind it).
__device__ __forceinline__ bool red_vec(const float* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Adds N sums (times scale) to p[0 .. N): a CTA's accumulator rows into the call's
// gradient, every CTA into the same addresses.  Lanes hold different rows, so a
// scalar add is one L2 operation for 4 bytes and 152 CTAs' worth of them took
// ~35 us at the end of a kernel; 16-byte reductions take a quarter of the operations
// (decoder training of 307,200 / 1,088,640 pixels 137 / 307 -> 101 / 271 us,
// smoothing of 1M Gaussians 442 -> 401 us).
template <int N>
__device__ __forceinline__ void red_row(float* p, const float* v, float scale, bool vec)
{
    if (vec) {
#pragma unroll
        for (int j = 0; j < N; j += 4)
            atomicAdd(reinterpret_cast<float4*>(p + j),
                      make_float4(v[j] * scale, v[j + 1] * scale, v[j + 2] * scale, v[j + 3] * scale));
    } else {
#pragma unroll
        for (int j = 0; j < N; ++j) atomicAdd(p + j, v[j] * scale);
    }
}

// v where the layer output h (16 columns at addr) is positive, else 0, as BF16 pairs.
__device__ __forceinline__ void relu_mask16(const float* v, uint32_t addr, uint32_t* w)
{
    uint32_t h[8];
    lds128(addr, h);
    lds128(addr + 128, h + 4);
    pack16(v, w);
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] &= positive2(h[j]);
}

// 8 floats -> 8 bf16 in one 16-byte shared store at a shared-memory address.
__device__ __forceinline__ void sts_bf16x8(uint32_t addr, const float* v)
{
    __nv_bfloat162 h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    const uint4 u = *reinterpret_cast<uint4*>(h);
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(u.x), "r"(u.y), "r"(u.z), "r"(u.w)
                 : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Hide a value's origin from the optimiser, so that what is derived from it is
// recomputed where used instead of being kept live across a loop.
__device__ __forceinline__ uint32_t opaque(uint32_t x)
{
    asm volatile("" : "+r"(x));
    return x;
}

// Fill rows [0,R) x cols [0,C) of a canonical buffer from fp32 row-major src
// (src[r*ld + c], zero outside [0,rs) x [0,cs)); all threads of the block.
__device__ __forceinline__ void sbuf_fill(const SBuf& b, int R, const float* src, int ld, int rs, int cs)
{
    const int chunks = R * (b.C >> 3);
    for (int i = threadIdx.x; i < chunks; i += blockDim.x) {
        const int r = i / (b.C >> 3), c0 = (i % (b.C >> 3)) * 8;
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (r < rs && c0 + j < cs) ? src[(size_t)r * ld + c0 + j] : 0.f;
        sbuf_store8(b, r, c0, v);
    }
}

// The same for a whole [R x C] matrix at a 16-byte aligned address, four 8-column
// pieces in flight per thread (a kernel's first microseconds are these loads).
__device__ __forceinline__ void sbuf_fill_rows(const SBuf& b, int R, const float* src)
{
    if (reinterpret_cast<uintptr_t>(src) & 15u) {
        sbuf_fill(b, R, src, b.C, R, b.C);
        return;
    }
    const int w = b.C >> 3, pieces = R * w;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    for (int i0 = threadIdx.x; i0 < pieces; i0 += 4 * blockDim.x) {
        float4 x[4][2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + q * blockDim.x;
            if (i < pieces) {
                x[q][0] = __ldg(s4 + 2 * i);
                x[q][1] = __ldg(s4 + 2 * i + 1);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + q * blockDim.x;
            if (i < pieces) sbuf_store8(b, i / w, (i % w) * 8, reinterpret_cast<const float*>(x[q]));
        }
    }
}

// Arrays that a call's kernels add into, cleared by one launch: a memset each costs
// 1-2 us on the stream (smoothing 100,000 Gaussians 95.5 -> 82.0 us with the wider
// weight loads, a training call at 8-128-256-128 on one tile 56.7 -> 46.6 us).
struct ZeroList {
    float* p[9];
    int n[9];
};

static __global__ void __launch_bounds__(256) zero_list_kernel(const ZeroList z)
{
    float* const p = z.p[blockIdx.x];
    const int n = z.n[blockIdx.x];
    for (int i = blockIdx.y * 256 + threadIdx.x; i < n; i += 256 * gridDim.y) p[i] = 0.f;
}

inline le_status zero_list(const ZeroList& z, int arrays, cudaStream_t s)
{
    zero_list_kernel<<<dim3(arrays, 8), 256, 0, s>>>(z);
    LE_LAUNCHED();
    return LE_OK;
}

// cuTensorMapEncodeTiled from the driver (once per process).
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline le_status tensor_map_encoder(EncodeTiled* fn)
{
    static EncodeTiled cached = nullptr;
    if (!cached) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &qr) !=
                cudaSuccess ||
            qr != cudaDriverEntryPointSuccess || !p) {
            set_error("cuTensorMapEncodeTiled is not available from the driver");
            return LE_ERR_CUDA;
        }
        cached = reinterpret_cast<EncodeTiled>(p);
    }
    *fn = cached;
    return LE_OK;
}

}  // namespace tc
}  // namespace leg
