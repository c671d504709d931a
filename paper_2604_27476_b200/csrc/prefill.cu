// Prompt processing for sm_100a: KV <- Prefill(x_1:T) (Eq. 3 of the paper).
//
// The T given tokens go through the layers together, so every projection is a dense [T x K] x [K x N] contraction:
//   * prefill_gemm_kernel: persistent, output tiles of 128 x 128 or 256.  A producer thread stages bf16 operand
//     tiles in shared memory by TMA (128-byte swizzle), one thread issues tcgen05.mma with the fp32 accumulator in tensor
//     memory, four warps read the accumulator back (tcgen05.ld) and apply the operator's epilogue:
//       QKV      : + bias, rotate-half RoPE of q and k, q to the work buffer, k and v rows to the cache;
//       O / down : added to the fp32 residual stream; the rows the next contraction reads (x * w, for the norm) with their sums of squares;
//       gate/up  : SwiGLU, silu(gate) * up, to the bf16 activation buffer.
//     RMSNorm's factor 1 / rms multiplies the results of QKV and gate/up instead of their operand rows.
//   * prefill_tile_kernel: the same contractions where the tiles fit the SMs in one round: clusters of CTAs share the K of a tile.
//   * prefill_attention_tc_kernel: causal attention of the T queries over the cache rows (prefix + the T new rows), also on
//     tcgen05: S = Q K^T and O = P V in tensor memory, online softmax by warps that own the rows (see the kernel).
//   * prefill_norm_kernel: embedding, and the norm behind a contraction that leaves K-split partial sums; one CTA per row.
// Every activation enters the tensor cores as TWO bf16 pieces (hi + lo, 16 mantissa bits; twice the multiplies, one load of
// the weight tile), because single bf16 activations put the logits of a 28-layer model outside the step's tolerance
// (measured: 3.6e-2 max-abs).  The residual stream stays fp32.
// Every wait on an mbarrier is bounded; a wait that runs out raises PrefillBuffers::error and the CTA drains and returns.
#include "prefill.h"

#include <cuda.h>
#include <cuda_bf16.h>

#include "tensor_map.h"

namespace edgefm {
namespace {

// ---- PTX wrappers ----------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `limit` polls or as soon as another thread of the CTA has given up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag, uint32_t limit) {
    for (uint32_t i = 0; i < limit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 63u && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// A CTA that gives up waits for what it has under way (copies into its shared memory, multiplies), in the end with a bound of its own.
constexpr uint32_t PF_LAND_POLLS = 1u << 24;
__device__ __forceinline__ void mbar_land(uint64_t *bar, uint32_t parity) {
#pragma unroll 1
    for (uint32_t i = 0; i < PF_LAND_POLLS && !mbar_try_wait(bar, parity); ++i) { }
}
// The copies of a ring: `issued` stages were asked for, the last `stages` of them may be on their way.  To be called behind a barrier that every
// wait of the CTA precedes: a producer that has sent for everything is done long before another thread's wait runs out.  extra_arrivals: the
// arrivals that nobody else makes (GemmArgs).  Not inlined: it hardly ever runs, and cost the clustered kernel up to 7 registers.
__device__ __noinline__ void ring_land(uint64_t *full_bar, int issued, int stages, uint32_t extra_arrivals) {
#pragma unroll 1
    for (int j = issued > stages ? issued - stages : 0; j < issued; ++j) {
        uint64_t *bar = full_bar + j % stages;
        for (uint32_t e = 0; e < extra_arrivals; ++e) mbar_arrive(bar);
        mbar_land(bar, (j / stages) & 1);
    }
}
// The same for a pair of CTAs, whose copies the first one counts: it has sent for `mine` stages and expected both CTAs' bytes for each, the second
// for `peers`.  Neither is more than a ring ahead (a stage is sent for again when the multiplies of both have read it), so every stage
// named here waits in its last phase.  What only one of them has sent for is put right: the first CTA expects the other's half, or counts the
// half that will not come as landed.
__device__ __forceinline__ void mbar_complete_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void pair_land(uint64_t *full_bar, int mine, int peers, int stages, uint32_t half_bytes, uint32_t extra_arrivals) {
    const int issued = mine > peers ? mine : peers;
#pragma unroll 1
    for (int j = issued > stages ? issued - stages : 0; j < issued; ++j) {
        if (j >= mine) mbar_expect_tx(full_bar + j % stages, half_bytes);
        else if (j >= peers) mbar_complete_tx(full_bar + j % stages, half_bytes);
    }
    ring_land(full_bar, issued, stages, extra_arrivals);
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
                     smem_u32(dst)),
                 "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
                 : "memory");
}

// Programmatic dependent launch: every kernel of the prefill chain lets its successor be launched as soon as all of its own CTAs
// have started (pdl_trigger), and touches what other kernels write only after its predecessor has completed and its writes are visible
// (pdl_wait).  What overlaps is the successor's launch and set-up (barriers, tensor memory, descriptor fetch, first weight tiles).  A kernel
// that allocates tensor memory triggers behind the allocation: several kernels may be resident on an SM at once, and one that waits for
// its predecessor must never hold the columns the predecessor still needs.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Descriptor fetch ahead of the first copy that uses the map (the map is a kernel parameter).
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]^T: 128 x N x 16, bf16 operands (both K-major), fp32 accumulator.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The same with the A operand in tensor memory (lane = row, 16-bit elements packed two per column, K along the columns).
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The same over a pair of CTAs (a cluster of two): 256 x N x 16, issued by the first.  Either CTA holds 128 rows of A, half of B's rows and
// its own rows of the accumulator, at the same places.
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// one arrival at the barrier of both CTAs when the pair's multiplies issued so far have finished
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                 "h"(static_cast<uint16_t>(3))
                 : "memory");
}
// a tile into this CTA's shared memory, its bytes counted at a barrier of the pair's first CTA (a shared::cluster address)
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
                     smem_u32(dst)),
                 "l"(map), "r"(x), "r"(y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// The mbarrier receives one arrival when every tcgen05.mma issued so far by this thread has finished.
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 32 lanes x 32 columns of fp32: thread i of the warp receives row (lane base + i), columns c .. c + 31.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v) {
    uint32_t *r = reinterpret_cast<uint32_t *>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, "
        "%18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float *v) {
    const uint32_t *r = reinterpret_cast<const uint32_t *>(v);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, "
        "%19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]),
        "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]),
        "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float *v) {
    const uint32_t *r = reinterpret_cast<const uint32_t *>(v);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]),
        "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// the values of a tmem_ld32 issued earlier are there (nothing that uses them moves above this)
__device__ __forceinline__ void tmem_ld_ready(float *v) {
    uint32_t *r = reinterpret_cast<uint32_t *>(v);
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]),
                   "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]),
                   "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]),
                   "+r"(r[31])::"memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major bf16 tile written by TMA with the 128-byte swizzle: rows of 64 elements
// (128 bytes), groups of 8 rows 1024 bytes apart.  Fields: start address >> 4 (bits 0-13), leading byte offset >> 4 (16-29;
// 1, unused with this swizzle), stride byte offset >> 4 (32-45) = 64, descriptor version 1 (46-47), layout 2 = 128-byte
// swizzle (61-63).  A step of 16 elements along K inside the 128-byte row adds 32 bytes to the start address.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr) {
    return static_cast<uint64_t>((smem_addr >> 4) & 0x3fffu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor: fp32 accumulator (bits 4-5 = 1), A and B bf16 (7-9 = 1, 10-12 = 1), both K-major (15, 16 = 0),
// N >> 3 (17-22), M >> 4 (24-28).
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(m >> 4) << 24);
}

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
    return static_cast<uint32_t>(f32_to_bf16_bits(lo)) | (static_cast<uint32_t>(f32_to_bf16_bits(hi)) << 16);
}

// An fp32 activation as two bf16 pieces, hi = bf16(x), lo = bf16(x - hi): 16 mantissa bits enter the tensor cores (the
// weights are bf16 exactly), so a contraction's operand rounding stays below 2^-17 relative.
__device__ __forceinline__ void split2(float x, uint16_t &hi, uint16_t &lo) {
    hi = f32_to_bf16_bits(x);
    lo = f32_to_bf16_bits(x - bf16_bits_to_f32(hi));
}
__device__ __forceinline__ void split2x2(float a, float b, uint32_t &hi, uint32_t &lo) {
    uint16_t ah, al, bh, bl;
    split2(a, ah, al);
    split2(b, bh, bl);
    hi = static_cast<uint32_t>(ah) | (static_cast<uint32_t>(bh) << 16);
    lo = static_cast<uint32_t>(al) | (static_cast<uint32_t>(bl) << 16);
}

// The same split by truncation (hi = the upper 16 bits of x, lo = the upper 16 bits of x - hi; x - hi is exact): no conversion
// instruction, which shares the special-function pipe with exp2 in the attention loop.  Error below 2^-16 relative.
__device__ __forceinline__ void split2x2_trunc(float a, float b, uint32_t &hi, uint32_t &lo) {
    const uint32_t ab = __float_as_uint(a), bb = __float_as_uint(b);
    hi = __byte_perm(ab, bb, 0x7632);
    const float ra = a - __uint_as_float(ab & 0xffff0000u), rb = b - __uint_as_float(bb & 0xffff0000u);
    lo = __byte_perm(__float_as_uint(ra), __float_as_uint(rb), 0x7632);
}

// ---- small kernels -----------------------------------------------------------------------------------------------------
// (cos, sin) of angle (position + t) * theta^(-2 j / d), evaluated in double and rounded once.
__global__ void __launch_bounds__(256) prefill_rope_kernel(float2 *rope, int n, int half, int position, double theta) {
    pdl_trigger();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * half) return;
    const int t = i / half, j = i % half;
    const double inv = pow(theta, -static_cast<double>(j) / static_cast<double>(half));
    double sn, cs;
    sincos(static_cast<double>(position + t) * inv, &sn, &cs);
    rope[i] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
}

// One CTA of 128 threads per row: y = x * rsqrt(mean(x^2) + eps) * w, stored as two bf16 planes (hi, lo; `plane` elements apart).  With `embed` the row is first fetched from the embedding
// table (bf16 -> fp32) and written to the residual stream.  Thread 0 of the grid also records the new cache length.
__global__ void __launch_bounds__(128) prefill_norm_kernel(float *resid, uint16_t *xn, size_t plane, const uint16_t *w, const uint16_t *embed,
                                                           const int *tokens, int n, int H, float eps, StepState *st, int new_len,
                                                           int new_pos, const float *part, int splits, size_t part_plane) {
    pdl_trigger();
    pdl_wait();
    if (st && blockIdx.x == 0 && threadIdx.x == 0) {
        st->cur_len = new_len;
        st->next_position = new_pos;
        if (st->status != STATUS_TIMEOUT) st->status = 0;
    }
    __shared__ float red[4];
    const int row = blockIdx.x, tid = threadIdx.x;
    float *x = resid + static_cast<size_t>(row) * H;
    uint16_t *y = xn + static_cast<size_t>(row) * H;
    // H is a multiple of 8: eight values per lane and round, 16- and 32-byte accesses
    const uint16_t *e = embed ? embed + static_cast<size_t>(tokens[row]) * H : nullptr;
    float ss = 0.f;
    for (int j = tid * 8; j < H; j += 1024) {
        float v[8];
        if (e) {
            const uint4 b = *reinterpret_cast<const uint4 *>(e + j);
            v[0] = bf16lo(b.x); v[1] = bf16hi(b.x); v[2] = bf16lo(b.y); v[3] = bf16hi(b.y);
            v[4] = bf16lo(b.z); v[5] = bf16hi(b.z); v[6] = bf16lo(b.w); v[7] = bf16hi(b.w);
            *reinterpret_cast<float4 *>(x + j) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4 *>(x + j + 4) = make_float4(v[4], v[5], v[6], v[7]);
        } else {
            const float4 a = *reinterpret_cast<const float4 *>(x + j), c = *reinterpret_cast<const float4 *>(x + j + 4);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = c.x; v[5] = c.y; v[6] = c.z; v[7] = c.w;
            if (splits > 1) {   // the K-split partial sums of the contraction before: added in plane order, written back
                for (int sp = 0; sp < splits; ++sp) {
                    const float *q = part + sp * part_plane + static_cast<size_t>(row) * H + j;
                    const float4 pa = *reinterpret_cast<const float4 *>(q), pc = *reinterpret_cast<const float4 *>(q + 4);
                    v[0] += pa.x; v[1] += pa.y; v[2] += pa.z; v[3] += pa.w; v[4] += pc.x; v[5] += pc.y; v[6] += pc.z; v[7] += pc.w;
                }
                *reinterpret_cast<float4 *>(x + j) = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4 *>(x + j + 4) = make_float4(v[4], v[5], v[6], v[7]);
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) ss = fmaf(v[i], v[i], ss);
    }
    ss = warp_sum(ss);
    if ((tid & 31) == 0) red[tid >> 5] = ss;
    __syncthreads();
    ss = (red[0] + red[1]) + (red[2] + red[3]);
    const float r = rsqrtf(ss / static_cast<float>(H) + eps);
    for (int j = tid * 8; j < H; j += 1024) {
        const float4 a = *reinterpret_cast<const float4 *>(x + j), c = *reinterpret_cast<const float4 *>(x + j + 4);
        const uint4 wb = *reinterpret_cast<const uint4 *>(w + j);
        uint4 hi, lo;
        split2x2(a.x * r * bf16lo(wb.x), a.y * r * bf16hi(wb.x), hi.x, lo.x);
        split2x2(a.z * r * bf16lo(wb.y), a.w * r * bf16hi(wb.y), hi.y, lo.y);
        split2x2(c.x * r * bf16lo(wb.z), c.y * r * bf16hi(wb.z), hi.z, lo.z);
        split2x2(c.z * r * bf16lo(wb.w), c.w * r * bf16hi(wb.w), hi.w, lo.w);
        *reinterpret_cast<uint4 *>(y + j) = hi;
        *reinterpret_cast<uint4 *>(y + plane + j) = lo;
    }
}

// Compressed cache (Sec. 3.9): one warp per new row (k rows, then v rows) of the fp32 staging buffers [nkv][stride / d][d];
// scale = amax / 127, code = clamp(rint(x * (127 / amax))) in fp32 -- the arithmetic of the decode step's own row.
__global__ void __launch_bounds__(256) prefill_quantize_rows_kernel(const float *k, const float *v, long long stage_stride, signed char *kc,
                                                                    signed char *vc, float *ks, float *vs, int nkv, int n, int d,
                                                                    int max_context, int slot0) {
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const long long r = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5, rows = static_cast<long long>(nkv) * n;
    if (r >= 2 * rows) return;
    const bool is_v = r >= rows;
    const long long rr = is_v ? r - rows : r;
    const int t = static_cast<int>(rr % n), g = static_cast<int>(rr / n);
    const float *src = (is_v ? v : k) + g * stage_stride + static_cast<long long>(t) * d;
    const long long row = static_cast<long long>(g) * max_context + slot0 + t;
    float x[4];                                                              // d <= 128: at most 4 values per lane
    float amax = 0.f;
    for (int e = 0; e < 4; ++e) {
        const int j = lane + 32 * e;
        x[e] = j < d ? src[j] : 0.f;
        amax = fmaxf(amax, fabsf(x[e]));
    }
    amax = warp_max(amax);
    const float inv = amax > 0.f ? __fdiv_rn(127.0f, amax) : 0.f;
    signed char *dst = (is_v ? vc : kc) + row * d;
    for (int e = 0; e < 4; ++e) {
        const int j = lane + 32 * e;
        if (j < d) dst[j] = static_cast<signed char>(static_cast<int>(fminf(fmaxf(rintf(__fmul_rn(x[e], inv)), -127.f), 127.f)));
    }
    if (lane == 0) (is_v ? vs : ks)[row] = amax > 0.f ? __fdiv_rn(amax, 127.0f) : 0.f;
}

// Output layer for ONE row (the prompt's last token): final RMSNorm, logits = W x over `rows` rows of the output matrix (bf16
// weights, fp32 x and sums), greedy token (larger value wins, equal values -> lower row), and the device state a decode step
// would leave.  A matrix-vector product: bound by the one pass over W.  grid: any; 256 threads; dynamic shared memory H floats.
constexpr int HEAD_CTAS_PER_SM = 3;   // 2: 16 warps an SM leave its loads idle between two groups of rows (2.6 TB/s where a row is 1792 bytes long)
__global__ void __launch_bounds__(256, HEAD_CTAS_PER_SM) prefill_head_kernel(const float *x, const uint16_t *wnorm, const uint16_t *lm, const int *ids, int rows,
                                                           int H, float eps, float *logits_out, int *next_token_out, float *part_val,
                                                           int *part_idx, unsigned *ticket, StepState *st, int token, int pos) {
    extern __shared__ __align__(16) float pf_xs[];
    __shared__ float red[8], bvs[8];
    __shared__ int bis[8], is_last;
    // four rows per round, two rounds of columns unrolled: 96 KB of loads in flight per SM (two rows, 16 KB: 2.6 TB/s)
    constexpr int R = 4;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, stride = gridDim.x * 8;
    pdl_trigger();
    for (int i = 0; i < R; ++i)          // the first round's rows are sent for to L2 while the predecessor still runs (nothing writes weights)
        if (const int r = blockIdx.x * 8 + warp + i * stride; r < rows)
            for (int j = lane * 64; j < H; j += 2048) asm volatile("prefetch.global.L2 [%0];" ::"l"(lm + static_cast<size_t>(r) * H + j));
    pdl_wait();
    float ss = 0.f;
    for (int j = tid; j < H; j += 256) ss = fmaf(x[j], x[j], ss);
    ss = warp_sum(ss);
    if (lane == 0) red[warp] = ss;
    __syncthreads();
    ss = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
    const float r = rsqrtf(ss / static_cast<float>(H) + eps);
    for (int j = tid; j < H; j += 256) pf_xs[j] = x[j] * r * bf16_bits_to_f32(wnorm[j]);
    __syncthreads();
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    for (int row = blockIdx.x * 8 + warp; row < rows; row += R * stride) {
        const uint16_t *w[R];
        float a[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int r = row + i * stride;
            w[i] = lm + static_cast<size_t>(r < rows ? r : row) * H;
            a[i] = 0.f;
        }
#pragma unroll 2
        for (int j = lane * 8; j < H; j += 256) {
            uint4 u[R];
#pragma unroll
            for (int i = 0; i < R; ++i) u[i] = __ldcs(reinterpret_cast<const uint4 *>(w[i] + j));
            const float4 x0 = *reinterpret_cast<const float4 *>(pf_xs + j), x1 = *reinterpret_cast<const float4 *>(pf_xs + j + 4);
#pragma unroll
            for (int i = 0; i < R; ++i) a[i] = dot8(u[i], x0, x1, a[i]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int r = row + i * stride;
            a[i] = warp_sum(a[i]);
            if (lane == 0 && r < rows) {
                if (logits_out) logits_out[r] = a[i];
                if (arg_better(a[i], r, bv, bi)) { bv = a[i]; bi = r; }
            }
        }
    }
    if (lane == 0) { bvs[warp] = bv; bis[warp] = bi; }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < 8; ++w)
            if (arg_better(bvs[w], bis[w], bv, bi)) { bv = bvs[w]; bi = bis[w]; }
        part_val[blockIdx.x] = bv;
        part_idx[blockIdx.x] = bi;
        __threadfence();
        is_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (is_last && warp == 0) {      // the last CTA to finish merges the CTAs' candidates
        __threadfence();
        bv = -INFINITY; bi = 0x7fffffff;
        for (int i = lane; i < static_cast<int>(gridDim.x); i += 32) {
            const float v = __ldcg(part_val + i);
            const int ix = __ldcg(part_idx + i);
            if (arg_better(v, ix, bv, bi)) { bv = v; bi = ix; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (arg_better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
        }
        if (lane == 0) {
            if (bi == 0x7fffffff) bi = 0;
            if (ids) bi = ids[bi];   // pruned vocabulary: row index -> token id
            if (next_token_out) *next_token_out = bi;
            st->token = token;
            st->position = pos;
            st->next_token = bi;
            st->next_position = pos + 1;
            st->n_accepted = 1;
            *ticket = 0u;
        }
    }
}

// Greedy tokens of the m <= PF_VERIFY_MAX rows of a logits matrix [m][rows] and the acceptance rule of a verified block (Sec. 3.11)
// on the device: proposal t + 1 is accepted if tokens[t + 1] equals the greedy token after token t, verification stops at the
// first mismatch; the cache length becomes slot0 + n_accepted (the rows behind it are overwritten later), the next token is the
// greedy token after the last accepted one.  The logits come from a contraction over the output matrix (EPI_LOGITS).
__global__ void __launch_bounds__(256) prefill_verify_pick_kernel(const float *logits, const int *ids, int rows, int m, const int *tokens,
                                                                  float *part_val, int *part_idx, unsigned *ticket, StepState *st, int slot0,
                                                                  int pos, int *n_accepted_out, int *next_token_out) {
    pdl_trigger();
    pdl_wait();
    __shared__ float bvs[8][PF_VERIFY_MAX];
    __shared__ int bis[8][PF_VERIFY_MAX], is_last;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int t = 0; t < m; ++t) {
        float bv = -INFINITY;
        int bi = 0x7fffffff;
        for (int r = blockIdx.x * 256 + tid; r < rows; r += gridDim.x * 256) {
            const float v = logits[static_cast<size_t>(t) * rows + r];
            if (arg_better(v, r, bv, bi)) { bv = v; bi = r; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (arg_better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
        }
        if (lane == 0) { bvs[warp][t] = bv; bis[warp][t] = bi; }
    }
    __syncthreads();
    if (tid < m) {
        float v = bvs[0][tid];
        int ix = bis[0][tid];
        for (int w = 1; w < 8; ++w)
            if (arg_better(bvs[w][tid], bis[w][tid], v, ix)) { v = bvs[w][tid]; ix = bis[w][tid]; }
        part_val[blockIdx.x * PF_VERIFY_MAX + tid] = v;
        part_idx[blockIdx.x * PF_VERIFY_MAX + tid] = ix;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) is_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (is_last && warp == 0) {
        __threadfence();
        int greedy = 0;
        if (lane < m) {
            float v = -INFINITY;
            int ix = 0x7fffffff;
            for (int i = 0; i < static_cast<int>(gridDim.x); ++i) {
                const float pv = __ldcg(part_val + i * PF_VERIFY_MAX + lane);
                const int pi = __ldcg(part_idx + i * PF_VERIFY_MAX + lane);
                if (arg_better(pv, pi, v, ix)) { v = pv; ix = pi; }
            }
            if (ix == 0x7fffffff) ix = 0;
            greedy = ids ? ids[ix] : ix;
        }
        int n_acc = 1, next = __shfl_sync(0xffffffffu, greedy, 0);
        for (int t = 1; t < m; ++t) {
            const int g_prev = __shfl_sync(0xffffffffu, greedy, t - 1), g_t = __shfl_sync(0xffffffffu, greedy, t);
            if (n_acc == t && tokens[t] == g_prev) { n_acc = t + 1; next = g_t; }
        }
        if (lane == 0) {
            if (next_token_out) *next_token_out = next;
            if (n_accepted_out) *n_accepted_out = n_acc;
            st->token = tokens[0];
            st->position = pos;
            st->next_token = next;
            st->next_position = pos + n_acc;
            st->cur_len = slot0 + n_acc;
            st->n_accepted = n_acc;
            *ticket = 0u;
        }
    }
}

// ---- the contraction -------------------------------------------------------------------------------------------------------
enum { EPI_QKV = 0, EPI_RESID = 1, EPI_SWIGLU = 2, EPI_LOGITS = 3 };   // EPI_LOGITS: plain fp32 store to g.resid [M][N] (output layer)

struct GemmArgs {
    int M, N, K;              // rows (tokens), output features (gate/up: F, each of gate and up), reduction length
    int *error;
    uint32_t wait_limit;      // polls a wait on an mbarrier may take
    uint32_t extra_arrivals;  // 0; 1 (tests): the stage barriers expect an arrival nobody makes, so the first wait runs out
    // RMSNorm of the operand rows, where the contraction before left x * w without the factor 1 / rms (a factor of the whole row, so it
    // may as well multiply the row's results): sums of squares of its pieces, [ss_pieces][ss_stride]; null = rows are normalised
    const float *ss_in;
    int ss_pieces;
    size_t ss_stride;
    float eps;
    // QKV
    const uint16_t *bias;     // [N] or null
    const float2 *rope;       // [M][d/2]
    uint16_t *q_out;          // [2][..][nq d]: hi and lo planes
    size_t q_plane;           // elements between the planes
    uint16_t *k_rows, *v_rows;  // the layer's cache at the first new slot: + head * head_stride + row * d
    float *k_stage, *v_stage;   // compressed cache: the rows go here in fp32 instead ([nkv][stage_stride / d rows][d]) and are
    long long stage_stride;     // compressed by prefill_quantize_rows_kernel
    int nq, nkv, d;
    long long head_stride;
    // O / down
    float *resid;             // [M][N]
    const uint16_t *norm_w;   // weights of the norm that follows, or null; then the epilogue also leaves
    uint16_t *xw;             // ... x * w of the new residual stream, [2][..][N]: hi and lo planes
    size_t x_plane;
    float *ss_out;            // ... and the sums of squares of its pieces (at most 64 columns of a tile), [piece][ss_stride]
    int splits;               // K split into this many units per output tile (1 = none).  With a split the units write their
    float *part;              // partial sums to part[split][..][N] (planes `part_plane` elements apart) instead of adding to resid;
    size_t part_plane;        // the norm kernel that follows adds the planes to the residual stream in a fixed order.
    // gate/up
    uint16_t *act;            // [2][..][N]: hi and lo planes
    size_t act_plane;
    int bn;                   // output columns of a tile: 64, 128 or 256; pairs that add to the residual stream: any multiple of 16 from 144 to 256
    // prefill_tile_kernel
    int cluster;              // CTAs that share the K of an output tile
    int a_rows;               // rows of an activation tile that are loaded (a multiple of 8, at most 128)
    int tmem_cols;            // tensor memory a CTA allocates (a power of two)
    int stages;
};

constexpr int PF_BM = 128, PF_BK = 64;
constexpr int PF_SPLIT_MAX = 8;               // K splits of a contraction that adds to the residual stream: up to 4, up to 8 when the
                                             // tokens fit one row tile (short prompts, verified blocks: the grids are smallest there)

// ---- epilogues: eight lanes take a row, four rows per warp and step -----------------------------------------------------------
// Accumulators come out of tensor memory a row per thread; stored like that, an instruction touches 32 lines (1.5B shape, 2048 tokens:
// O took 43 us and the norm behind it 6, now 29 together; QKV 37, now 33).  So a chunk of 64 accumulator columns passes through
// shared memory, and a lane then holds four consecutive columns of each of the chunk's two 32-column halves (a, b): 64 to 128 bytes of
// a row per eight lanes.  The halves are the pairs an operator needs together: gate and up, or the two halves of a rotated head.
template <int EPI, int N_STEP> __device__ __forceinline__ void chunk_halves(int chunk, int d, int &a, int &b) {
    if (EPI == EPI_SWIGLU) { a = 32 * chunk; b = N_STEP + 32 * chunk; }
    else if (EPI == EPI_QKV && d == 128) { a = (chunk >> 1) * 128 + (chunk & 1) * 32; b = a + 64; }
    else { a = 64 * chunk; b = a + 32; }
}
// what a lane needs besides the accumulators: of its columns (biases, norm weights), and of a row and its columns (residuals, rotation)
struct ColVals { uint2 a, b; };
struct RowVals { float4 a, b; };

template <int EPI> __device__ __forceinline__ ColVals load_cols(const GemmArgs &g, int col_a, int col_b) {
    ColVals c{make_uint2(0u, 0u), make_uint2(0u, 0u)};
    const uint16_t *v = EPI == EPI_QKV ? g.bias : EPI == EPI_RESID ? g.norm_w : nullptr;
    if (v && col_a < g.N) c.a = *reinterpret_cast<const uint2 *>(v + col_a);
    if (v && col_b < g.N) c.b = *reinterpret_cast<const uint2 *>(v + col_b);
    return c;
}
template <int EPI> __device__ __forceinline__ RowVals load_row(const GemmArgs &g, int row, int col_a, int col_b) {
    RowVals r;
    r.a = r.b = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row >= g.M) return r;
    if (EPI == EPI_RESID && g.splits == 1) {
        const float *p = g.resid + static_cast<size_t>(row) * g.N;
        if (col_a < g.N) r.a = *reinterpret_cast<const float4 *>(p + col_a);
        if (col_b < g.N) r.b = *reinterpret_cast<const float4 *>(p + col_b);
    } else if (EPI == EPI_QKV && col_a < (g.nq + g.nkv) * g.d) {          // (cos, sin) of four pairs
        const float4 *p = reinterpret_cast<const float4 *>(g.rope + static_cast<size_t>(row) * (g.d >> 1) + (col_a & (g.d - 1)));
        r.a = p[0];
        r.b = p[1];
    }
    return r;
}
__device__ __forceinline__ void store_split4(uint16_t *p, size_t plane, const float *v) {
    uint2 hi, lo;
    split2x2(v[0], v[1], hi.x, lo.x);
    split2x2(v[2], v[3], hi.y, lo.y);
    *reinterpret_cast<uint2 *>(p) = hi;
    *reinterpret_cast<uint2 *>(p + plane) = lo;
}
__device__ __forceinline__ uint2 pack4_bf16(const float *v) { return make_uint2(pack2_bf16(v[0], v[1]), pack2_bf16(v[2], v[3])); }
__device__ __forceinline__ void unpack4(uint2 u, float *v) { v[0] = bf16lo(u.x); v[1] = bf16hi(u.x); v[2] = bf16lo(u.y); v[3] = bf16hi(u.y); }

// A lane's eight results of one row (output columns col_a .. col_a + 3 and col_b .. col_b + 3; gate/up: column col_a of both).  rs: 1 / rms
// of the operand row.  Returns the lane's share of the row's sum of squares (EPI_RESID with norm_w).
template <int EPI>
__device__ __forceinline__ float finish_row(const GemmArgs &g, int row, int col_a, int col_b, float4 va, float4 vb, const ColVals &cv,
                                            const RowVals &rv, float rs, int split) {
    float a[4] = {va.x, va.y, va.z, va.w}, b[4] = {vb.x, vb.y, vb.z, vb.w}, ss = 0.f;
    if (row >= g.M) return ss;
    if constexpr (EPI == EPI_RESID) {
        if (g.splits > 1) {              // a partial sum: added to the stream by the norm kernel
            float *p = g.part + split * g.part_plane + static_cast<size_t>(row) * g.N;
            if (col_a < g.N) *reinterpret_cast<float4 *>(p + col_a) = va;
            if (col_b < g.N) *reinterpret_cast<float4 *>(p + col_b) = vb;
            return ss;
        }
        auto half = [&](float *v, float4 r, uint2 w4, int col) {
            if (col >= g.N) return;
            v[0] += r.x; v[1] += r.y; v[2] += r.z; v[3] += r.w;
            *reinterpret_cast<float4 *>(g.resid + static_cast<size_t>(row) * g.N + col) = make_float4(v[0], v[1], v[2], v[3]);
            if (!g.norm_w) return;
            float w[4];
            unpack4(w4, w);
#pragma unroll
            for (int i = 0; i < 4; ++i) { ss = fmaf(v[i], v[i], ss); w[i] *= v[i]; }
            store_split4(g.xw + static_cast<size_t>(row) * g.N + col, g.x_plane, w);
        };
        half(a, rv.a, cv.a, col_a);
        half(b, rv.b, cv.b, col_b);
    } else if constexpr (EPI == EPI_LOGITS) {   // N need not be a multiple of 4 (a pruned vocabulary): scalar stores
        float *p = g.resid + static_cast<size_t>(row) * g.N;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (col_a + i < g.N) p[col_a + i] = a[i];
            if (col_b + i < g.N) p[col_b + i] = b[i];
        }
    } else if constexpr (EPI == EPI_SWIGLU) {
        if (col_a < g.N) {
            float o[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float gate = a[i] * rs, up = b[i] * rs;
                o[i] = gate / (1.f + __expf(-gate)) * up;
            }
            store_split4(g.act + static_cast<size_t>(row) * g.N + col_a, g.act_plane, o);
        }
    } else {                             // EPI_QKV: the chunk's halves are the two halves of (32 pairs of) a head; N is whole heads
        float ba[4], bb[4];
        unpack4(cv.a, ba);
        unpack4(cv.b, bb);
#pragma unroll
        for (int i = 0; i < 4; ++i) { a[i] = fmaf(a[i], rs, ba[i]); b[i] = fmaf(b[i], rs, bb[i]); }
        const int head = col_a / g.d, j = col_a & (g.d - 1), jb = j + (col_b - col_a);
        if (head < g.nq + g.nkv) {       // q or k: rotate-half pairs (j, j + d/2)
            const float c[4] = {rv.a.x, rv.a.z, rv.b.x, rv.b.z}, s[4] = {rv.a.y, rv.a.w, rv.b.y, rv.b.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float x = a[i], y = b[i];
                a[i] = x * c[i] - y * s[i];
                b[i] = y * c[i] + x * s[i];
            }
            if (head < g.nq) {           // queries keep both pieces
                uint16_t *dst = g.q_out + static_cast<size_t>(row) * g.nq * g.d + static_cast<size_t>(head) * g.d;
                store_split4(dst + j, g.q_plane, a);
                store_split4(dst + jb, g.q_plane, b);
                return ss;
            }
        }
        const bool is_v = head >= g.nq + g.nkv;
        const int hk = head - g.nq - (is_v ? g.nkv : 0);
        if (float *f = is_v ? g.v_stage : g.k_stage) {   // compressed cache: fp32 rows for the quantiser
            f += hk * g.stage_stride + static_cast<size_t>(row) * g.d;
            *reinterpret_cast<float4 *>(f + j) = make_float4(a[0], a[1], a[2], a[3]);
            *reinterpret_cast<float4 *>(f + jb) = make_float4(b[0], b[1], b[2], b[3]);
        } else {
            uint16_t *dst = (is_v ? g.v_rows : g.k_rows) + hk * g.head_stride + static_cast<size_t>(row) * g.d;
            *reinterpret_cast<uint2 *>(dst + j) = pack4_bf16(a);
            *reinterpret_cast<uint2 *>(dst + jb) = pack4_bf16(b);
        }
    }
    return ss;
}
// 1 / rms of an operand row from the sums of squares of its pieces
__device__ __forceinline__ float row_scale(const GemmArgs &g, int row) {
    if (!g.ss_in || row >= g.M) return 1.f;
    float ss = 0.f;
#pragma unroll 4
    for (int t = 0; t < g.ss_pieces; ++t) ss += g.ss_in[t * g.ss_stride + row];
    return rsqrtf(ss / static_cast<float>(g.K) + g.eps);
}
// the sum over the eight lanes of a row, stored by the first of them
__device__ __forceinline__ void store_row_ss(const GemmArgs &g, float ss, int row, int piece, int lane) {
    ss += __shfl_xor_sync(0xffffffffu, ss, 1);
    ss += __shfl_xor_sync(0xffffffffu, ss, 2);
    ss += __shfl_xor_sync(0xffffffffu, ss, 4);
    if ((lane & 7) == 0 && row < g.M) g.ss_out[piece * g.ss_stride + row] = ss;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, int rank) {   // the same place in the shared memory of another CTA of the cluster
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ int cluster_ld1(uint32_t addr) {
    int v;
    asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_st1(uint32_t addr, int v) { asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }

// COLUMNS of a tile.  128: 4 stages of 48 KB.  256: 3 stages of 64 KB, per k-block
// 64 KB of operands feed twice the multiplies of a narrow tile's 48 KB, which matters because operand delivery from L2, not
// the tensor pipe, bounds the narrow tiles.  Gate/up runs wide: 128 gate columns and their 128 up partners.
// PAIR: two row tiles, one in either CTA of a cluster of two, multiplied together (cta_group::2): a CTA fetches half of the weight tile only,
// 48 KB per k-block instead of 64, which leaves room for a fourth stage (gate/up and QKV by single CTAs, the rest by pairs: 4200 tokens, 7B
// shape, 97.2 ms, all by pairs 94.8; 1000 tokens, 3B, 12.60 and 12.43; these passes run into the power limit).
// The kernel is persistent (one CTA per SM, tiles dealt round-robin, neighbours sharing a weight tile) with TWO accumulators
// in tensor memory, so that the epilogue of a tile runs under the main loop of the next.
template <int COLUMNS, bool PAIR> struct GemmCfg {
    static constexpr int BN = COLUMNS;
    static constexpr int STAGES = COLUMNS == 256 && !PAIR ? 3 : 4;
    static constexpr int A_BYTES = PF_BM * PF_BK * 2, B_BYTES = BN * PF_BK * 2 / (PAIR ? 2 : 1);
    static constexpr int STAGE_BYTES = 2 * A_BYTES + B_BYTES;          // A hi, A lo, B
    static constexpr int CHUNK_BYTES = PF_BM * 64 * 4;                 // the epilogue's chunk of 64 columns
    static constexpr int SMEM = STAGES * STAGE_BYTES + CHUNK_BYTES + 1024;   // + room to align the first stage to 1024 bytes
};

template <int EPI, int COLUMNS, bool PAIR>
__global__ void __launch_bounds__(192) prefill_gemm_kernel(const __grid_constant__ CUtensorMap map_a_hi,
                                                           const __grid_constant__ CUtensorMap map_a_lo,
                                                           const __grid_constant__ CUtensorMap map_b, const GemmArgs g) {
    using C = GemmCfg<COLUMNS, PAIR>;
    static_assert(!PAIR || COLUMNS == 256, "a CTA of a pair fetches 128 of the 256 columns");
    const int BN = PAIR && EPI == EPI_RESID ? g.bn : C::BN;
    const int N_STEP = EPI == EPI_SWIGLU ? C::BN / 2 : BN;          // output columns (of g.N) a tile covers
    constexpr int CTAS = PAIR ? 2 : 1, TILE_M = CTAS * PF_BM;
    extern __shared__ uint8_t pf_dyn[];
    __shared__ uint64_t full_bar[C::STAGES], empty_bar[C::STAGES], acc_full[2], acc_empty[2], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, issued_sm, drained_sm;   // stages this CTA's producer has sent for; 1: its issuer has given up (drain_bar has an arrival)
    uint8_t *tiles = pf_dyn + ((1024u - (smem_u32(pf_dyn) & 1023u)) & 1023u);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = PAIR ? blockIdx.x & 1 : 0, worker = blockIdx.x / CTAS, workers = gridDim.x / CTAS;
    const int m_tiles = (g.M + TILE_M - 1) / TILE_M, n_tiles = (g.N + N_STEP - 1) / N_STEP;
    const int KB = (g.K + PF_BK - 1) / PF_BK;
    const int splits = EPI == EPI_RESID ? g.splits : 1;
    const int my_tiles = (m_tiles * n_tiles * splits - worker + workers - 1) / workers;
    // unit u of the grid-wide list: row tile u % m_tiles (neighbours share a weight tile), then the K split, then the column tile
    auto unit_of = [&](int i, int &m0, int &n0, int &kb0, int &kb1) {
        const int u = worker + i * workers, rest = u / m_tiles, sp = rest % splits;
        m0 = (u % m_tiles) * TILE_M + rank * PF_BM;
        n0 = (rest / splits) * N_STEP;
        kb0 = sp * KB / splits;
        kb1 = (sp + 1) * KB / splits;
        return sp;
    };

    if (threadIdx.x == 0) {
        prefetch_map(&map_a_hi); prefetch_map(&map_a_lo); prefetch_map(&map_b);
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(&full_bar[s], 1 + g.extra_arrivals); mbar_init(&empty_bar[s], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 4 * CTAS); }
        mbar_init(&drain_bar, 1);
        abort_flag = drained_sm = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {   // two accumulators: 2 BN columns of tensor memory, 128 lanes
        if constexpr (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(2 * C::BN) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(2 * C::BN) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    if constexpr (PAIR) cluster_sync(); else __syncthreads();   // a pair: the peer's barriers and tensor memory are there, too
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_trigger();   // (behind the allocation: see pdl_trigger)

    if (warp == 0 && lane == 0) {            // producer: operand tiles by TMA; a pair's bytes are counted by its first CTA
        bool ok = true;
        int issued = 0, m0, n0, kb0, kb1;
        auto load_b = [&](int kb, int s) {
            uint8_t *b = tiles + s * C::STAGE_BYTES + 2 * C::A_BYTES;
            if (rank == 0) mbar_expect_tx(&full_bar[s], PAIR ? 2 * (2 * C::A_BYTES + BN * PF_BK) : C::STAGE_BYTES);
            if constexpr (PAIR) {
                // B's rows: the first half here, the others in the peer (gate/up: the gate columns, the up columns)
                tma_load_2d_pair(b, &map_b, kb * PF_BK, n0 + rank * (EPI == EPI_SWIGLU ? g.N : BN / 2), cluster_addr(smem_u32(&full_bar[s]), 0));
            } else {
                tma_load_2d(b, &map_b, kb * PF_BK, n0, &full_bar[s]);
                if (EPI == EPI_SWIGLU) tma_load_2d(b + N_STEP * PF_BK * 2, &map_b, kb * PF_BK, g.N + n0, &full_bar[s]);
                else if (C::BN == 256) tma_load_2d(b + 128 * PF_BK * 2, &map_b, kb * PF_BK, 128 + n0, &full_bar[s]);
            }
        };
        auto load_a = [&](int kb, int s) {
            uint8_t *a = tiles + s * C::STAGE_BYTES;
            if constexpr (PAIR) {
                const uint32_t bar = cluster_addr(smem_u32(&full_bar[s]), 0);
                tma_load_2d_pair(a, &map_a_hi, kb * PF_BK, m0, bar);
                tma_load_2d_pair(a + C::A_BYTES, &map_a_lo, kb * PF_BK, m0, bar);
            } else {
                tma_load_2d(a, &map_a_hi, kb * PF_BK, m0, &full_bar[s]);
                tma_load_2d(a + C::A_BYTES, &map_a_lo, kb * PF_BK, m0, &full_bar[s]);
            }
        };
        // the weight tiles of the first stages before the predecessor is waited for, the output matrix is a weight, too (271 tokens behind 1000,
        // 1.5B shape: 3596 -> 3578 us a prompt)
        unit_of(0, m0, n0, kb0, kb1);
        const int first = my_tiles > 0 ? min(C::STAGES, kb1 - kb0) : 0;
        for (int it = 0; it < first; ++it) load_b(kb0 + it, it);
        pdl_wait();      // from here on the kernel reads what its predecessor wrote
        for (int i = 0, it = 0; i < my_tiles && ok; ++i) {
          unit_of(i, m0, n0, kb0, kb1);
          for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const int s = it % C::STAGES;
            if (it >= first) {
                if (it >= C::STAGES && !mbar_wait(&empty_bar[s], ((it / C::STAGES) - 1) & 1, &abort_flag, g.wait_limit)) { ok = false; break; }
                load_b(kb, s);
            }
            load_a(kb, s);
            issued = it + 1;
          }
        }
        issued_sm = issued;
    } else if (warp == 1 && lane == 0) {     // issuer (of a pair, the first CTA's): per stage 4 tcgen05.mma (K = 16 each) for the hi pieces, 4 for the lo pieces
        const uint32_t idesc = umma_idesc_bf16(TILE_M, BN);
        auto mma = [&](uint32_t acc, uint64_t da, uint64_t db, uint32_t accumulate) {
            if constexpr (PAIR) umma_bf16_pair(acc, da, db, idesc, accumulate); else umma_bf16(acc, da, db, idesc, accumulate);
        };
        auto commit = [&](uint64_t *bar) { if constexpr (PAIR) umma_commit_pair(bar); else umma_commit(bar); };
        pdl_wait();
        bool ok = true;
        for (int i = 0, it = 0; i < (rank == 0 ? my_tiles : 0) && ok; ++i) {
          const int buf = i & 1;
          const uint32_t acc = tmem + buf * C::BN;
          if (i >= 2) ok = mbar_wait(&acc_empty[buf], ((i >> 1) - 1) & 1, &abort_flag, g.wait_limit);   // its epilogue has read it
          if (!ok) break;
          tc_fence_after();
          int m0, n0, kb0, kb1;
          unit_of(i, m0, n0, kb0, kb1);
          for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const int s = it % C::STAGES;
            ok = mbar_wait(&full_bar[s], (it / C::STAGES) & 1, &abort_flag, g.wait_limit);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a = smem_u32(tiles + s * C::STAGE_BYTES), b = a + 2 * C::A_BYTES;
            const uint64_t da = umma_desc_sw128(a), dl = umma_desc_sw128(a + C::A_BYTES), db = umma_desc_sw128(b);
#pragma unroll
            for (int k = 0; k < PF_BK / 16; ++k) mma(acc, da + 2 * k, db + 2 * k, ((kb - kb0) | k) != 0);
#pragma unroll
            for (int k = 0; k < PF_BK / 16; ++k) mma(acc, dl + 2 * k, db + 2 * k, 1);
            commit(&empty_bar[s]);           // the stage is free again when these have read it
          }
          if (ok) commit(&acc_full[buf]);
        }
        if (!ok) {          // giving up: the multiplies already issued must finish before the tensor memory is freed
            commit(&drain_bar);
            mbar_land(&drain_bar, 0);
            drained_sm = 1;
        }
    } else if (warp >= 2) {                  // epilogue: warp w may read lanes 32 (w % 4) .. + 31 of tensor memory
      const int quarter = warp & 3, sub = lane >> 3, c8 = lane & 7;
      float4 *chunk = reinterpret_cast<float4 *>(tiles + C::STAGES * C::STAGE_BYTES) + quarter * 32 * 16;   // this warp's 32 rows x 64 columns
      pdl_wait();
      for (int i = 0; i < my_tiles; ++i) {
        int m0, n0, kb0, kb1;
        const int sp = unit_of(i, m0, n0, kb0, kb1), buf = i & 1;
        const float rs_own = EPI == EPI_QKV || EPI == EPI_SWIGLU ? row_scale(g, m0 + quarter * 32 + lane) : 1.f;
        const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (i >> 1) & 1, &abort_flag, g.wait_limit));   // warp-uniform: tcgen05.ld is .aligned
        if (!ok) break;
        tc_fence_after();
        const uint32_t trow = tmem + buf * C::BN + (static_cast<uint32_t>(quarter * 32) << 16);
        for (int ch = 0; ch < (BN + 63) / 64; ++ch) {
            int ca, cb;
            chunk_halves<EPI, EPI == EPI_SWIGLU ? C::BN / 2 : C::BN>(ch, g.d, ca, cb);
            if (n0 + ca >= g.N) break;
            int col_a = n0 + ca + 4 * c8, col_b = n0 + cb + 4 * c8;
            if (PAIR && EPI == EPI_RESID) {          // the last chunk may reach past the tile
                if (ca + 4 * c8 >= BN) col_a = g.N;
                if (cb + 4 * c8 >= BN) col_b = g.N;
            }
            const ColVals cv = load_cols<EPI>(g, col_a, col_b);
            RowVals rv[8];
            if constexpr (EPI == EPI_QKV || EPI == EPI_RESID) {
#pragma unroll
                for (int q = 0; q < 8; ++q) rv[q] = load_row<EPI>(g, m0 + quarter * 32 + 4 * q + sub, col_a, col_b);
            }
            __syncwarp();                    // the chunk before has been read
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) { // 16-byte pieces of a row, their index xor the row: no bank conflicts either way
                float v[32];
                tmem_ld32(trow + (hf ? cb : ca), v);
                tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    chunk[lane * 16 + ((hf * 8 + q) ^ (lane & 7))] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int r = 4 * q + sub, row = m0 + quarter * 32 + r;
                const float4 va = chunk[r * 16 + (c8 ^ (r & 7))], vb = chunk[r * 16 + 8 + (c8 ^ (r & 7))];
                const float rs = __shfl_sync(0xffffffffu, rs_own, r);
                const float ss = finish_row<EPI>(g, row, col_a, col_b, va, vb, cv, rv[q], rs, sp);
                if (EPI == EPI_RESID && g.norm_w && g.splits == 1) store_row_ss(g, ss, row, n0 / BN * ((BN + 63) / 64) + ch, lane);
            }
        }
        tc_fence_before();           // the accumulator may be overwritten: this warp has read its quarter
        __syncwarp();
        if (lane == 0) {
            if (rank == 0) mbar_arrive(&acc_empty[buf]); else mbar_arrive_remote(cluster_addr(smem_u32(&acc_empty[buf]), 0));
        }
      }
    }
    tc_fence_before();
    __syncwarp();
    if constexpr (PAIR) {                    // a pair leaves together: the first CTA's multiplies use both; it gives up together, too
        const uint32_t peer_abort = cluster_addr(smem_u32(&abort_flag), rank ^ 1);
        if (abort_flag) cluster_st1(peer_abort, 1);
        cluster_sync();
        if (abort_flag) {
            if (threadIdx.x == 0) {
                const int peers = cluster_ld1(cluster_addr(smem_u32(&issued_sm), rank ^ 1));
                if (rank == 0) pair_land(full_bar, issued_sm, peers, C::STAGES, 2 * C::A_BYTES + BN * PF_BK, g.extra_arrivals);
                else if (cluster_ld1(cluster_addr(smem_u32(&drained_sm), 0))) mbar_land(&drain_bar, 0);   // the first CTA's commit arrives here, too
            }
            cluster_sync();
        }
    } else {
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * C::BN) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * C::BN) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) {        // the CTA's shared memory is released when this thread leaves
        if (!PAIR) ring_land(full_bar, issued_sm, C::STAGES, g.extra_arrivals);
        atomicExch(g.error, 1);
    }
}

// The same contraction where the tiles fit the SMs in one round (short prompts): a cluster of g.cluster CTAs shares the K of one output
// tile, the partial tiles meet through distributed shared memory, every CTA finishes its share of the rows (77 tokens behind 1024, 0.5B
// shape: 1882 us a prompt by the persistent kernel and its K splits, 1438 so; 9 behind 2048, 1.5B: 2744 and 1799).  Such a pass is a
// chain of latencies, so everything here shortens the chain:
//   * tiles of half the columns where those fit the round, too: 64, or 64 + 64 for gate/up;
//   * the K of a tile is spread over up to eight SMs, and no partial sums pass through global memory and a kernel of their own;
//   * the weight tiles of the first stages are requested, the rest of this CTA's weights sent for to L2, BEFORE the predecessor is
//     waited for (nothing writes weights);
//   * at most 110 KB of shared memory where a CTA has few k-blocks and a partial tile that is no larger: two CTAs per SM, so that the successor's set-up and first weights overlap
//     this kernel's end; twice that where it has many (two stages of 48 KB: 27 us for 35 k-blocks, 1.8 MB, of a down projection);
//   * an activation tile is loaded without its idle rows (a multiple of 8; the multiplies read whatever lies behind it, for rows nobody
//     looks at);
//   * SWAP, up to 256 tokens: the weights are the 128 rows of the multiply and the tokens its columns.  Two row tiles then share one weight
//     tile, and idle rows cost nothing.  Where the tokens (padded to 8) are fewer than the tile's columns the hi and lo pieces lie side by
//     side, so that four multiplies of 2 x tokens columns take the place of eight of the tile's width
//     over 128 rows (which for 9 tokens, 1.5B shape, are 6.3 us of multiplies in a gate/up tile, by arithmetic: more than its weights take).
constexpr int TILE_STAGES_MAX = 8, TILE_THREADS = 256, TILE_SMEM = 110 * 1024, TILE_SMEM_DEEP = 220 * 1024, TILE_AHEAD = 32;

__device__ __forceinline__ float4 cluster_ld4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void prefetch_tile_l2(const CUtensorMap *map, int x, int y) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(map), "r"(x), "r"(y) : "memory");
}

template <int EPI, int BN, bool SWAP>
__global__ void __launch_bounds__(TILE_THREADS, 2) prefill_tile_kernel(const __grid_constant__ CUtensorMap map_a_hi,
                                                                       const __grid_constant__ CUtensorMap map_a_lo,
                                                                       const __grid_constant__ CUtensorMap map_b, const GemmArgs g) {
    constexpr int ROWS = SWAP ? 2 * PF_BM : PF_BM;       // of a tile at most
    constexpr int N_STEP = EPI == EPI_SWIGLU ? BN / 2 : BN, B_PARTS = EPI == EPI_SWIGLU || BN == 256 ? 2 : 1, CHUNKS = BN / 64;
    extern __shared__ uint8_t pf_dyn[];
    __shared__ uint64_t full_bar[TILE_STAGES_MAX], empty_bar[TILE_STAGES_MAX], acc_full, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, issued_sm;
    __shared__ float rs_sm[ROWS];
    uint8_t *tiles = pf_dyn + ((1024u - (smem_u32(pf_dyn) & 1023u)) & 1023u);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = g.cluster, tile = blockIdx.x / S, rank = blockIdx.x - tile * S, KB = (g.K + PF_BK - 1) / PF_BK;
    const int m_tiles = (g.M + ROWS - 1) / ROWS, n_tile = tile / m_tiles, m0 = (tile - n_tile * m_tiles) * ROWS, n0 = n_tile * N_STEP;
    const int kb0 = rank * KB / S, nkb = (rank + 1) * KB / S - kb0;
    const int a_bytes = g.a_rows * PF_BK * 2, stage_bytes = 2 * a_bytes + BN * PF_BK * 2;
    const int live = min(ROWS, g.M - m0), r0 = rank * live / S, r1 = (rank + 1) * live / S;   // rows of the tile; those this CTA finishes

    if (threadIdx.x == 0) {
        prefetch_map(&map_b); prefetch_map(&map_a_hi); prefetch_map(&map_a_lo);
#pragma unroll 1
        for (int s = 0; s < g.stages; ++s) { mbar_init(&full_bar[s], 1 + g.extra_arrivals); mbar_init(&empty_bar[s], 1); }
        mbar_init(&acc_full, 1);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_trigger();

    if (warp == 0 && lane == 0) {            // producer
        const int first = min(nkb, g.stages);
        // it: k-block of this CTA; what: 0 = its weight tile into stage s, 1 = asked for from memory only
        auto load_b = [&](int it, int s, bool into) {
            const int x = (kb0 + it) * PF_BK;
            uint8_t *b = tiles + s * stage_bytes + 2 * a_bytes;
            if (into) mbar_expect_tx(&full_bar[s], stage_bytes);
#pragma unroll
            for (int part = 0; part < B_PARTS; ++part) {     // gate and up, or 128 and 128 columns
                const int y = n0 + part * (EPI == EPI_SWIGLU ? g.N : 128);
                if (into) tma_load_2d(b + part * (BN * PF_BK * 2 / B_PARTS), &map_b, x, y, &full_bar[s]);
                else prefetch_tile_l2(&map_b, x, y);
            }
        };
        auto load_a = [&](int it, int s) {
            uint8_t *a = tiles + s * stage_bytes;
            tma_load_2d(a, &map_a_hi, (kb0 + it) * PF_BK, m0, &full_bar[s]);
            tma_load_2d(a + a_bytes, &map_a_lo, (kb0 + it) * PF_BK, m0, &full_bar[s]);
        };
        const int ahead = m0 == 0 ? min(nkb, first + TILE_AHEAD) : first;
#pragma unroll 1
        for (int it = 0; it < ahead; ++it) load_b(it, it, it < first);
        pdl_wait();
        int it = 0;
#pragma unroll 1
        for (int s = 0, phase = 1; it < nkb; ++it) {      // from the second round on: the stage is free when its multiplies are done
            if (it >= first) {
                if (!mbar_wait(&empty_bar[s], phase, &abort_flag, g.wait_limit)) break;
                load_b(it, s, true);
            }
            load_a(it, s);
            if (++s == g.stages) { s = 0; phase ^= 1; }
        }
        issued_sm = it;
    } else if (warp == 1 && lane == 0) {     // issuer
        pdl_wait();
        const bool side = 2 * g.a_rows <= 256;            // SWAP: hi and lo columns side by side (more do not fit one multiply)
        const uint32_t idesc = umma_idesc_bf16(PF_BM, !SWAP ? BN : side ? 2 * g.a_rows : g.a_rows);
        bool ok = true;
#pragma unroll 1
        for (int it = 0, s = 0, phase = 0; it < nkb; ++it) {
            ok = mbar_wait(&full_bar[s], phase, &abort_flag, g.wait_limit);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a = smem_u32(tiles + s * stage_bytes);
            const uint64_t da = umma_desc_sw128(a), db = umma_desc_sw128(a + 2 * a_bytes);
            if constexpr (SWAP) {            // (the lo rows lie right behind the hi rows)
#pragma unroll
                for (int k = 0; k < PF_BK / 16; ++k) umma_bf16(tmem, db + 2 * k, da + 2 * k, idesc, (it | k) != 0);
                if (!side) {
                    const uint64_t dl = umma_desc_sw128(a + a_bytes);
#pragma unroll
                    for (int k = 0; k < PF_BK / 16; ++k) umma_bf16(tmem, db + 2 * k, dl + 2 * k, idesc, 1);
                }
            } else {
                const uint64_t dl = umma_desc_sw128(a + a_bytes);
#pragma unroll
                for (int k = 0; k < PF_BK / 16; ++k) umma_bf16(tmem, da + 2 * k, db + 2 * k, idesc, (it | k) != 0);
#pragma unroll
                for (int k = 0; k < PF_BK / 16; ++k) umma_bf16(tmem, dl + 2 * k, db + 2 * k, idesc, 1);
            }
            umma_commit(&empty_bar[s]);
            if (++s == g.stages) { s = 0; phase ^= 1; }
        }
        umma_commit(ok ? &acc_full : &drain_bar);
        if (!ok) mbar_land(&drain_bar, 0);   // giving up: the multiplies already issued must finish before the tensor memory is freed
    }
    __syncwarp();
    pdl_wait();
    if ((warp & 6) == 2 && EPI != EPI_RESID)        // the scales of this CTA's rows
        for (int r = r0 + threadIdx.x - 64; r < r1; r += 64) rs_sm[r] = row_scale(g, m0 + r);

    // Steps of the epilogue, a warp each: row group (4 rows) item / chunks, chunk item % chunks.  The first step's vectors are fetched under
    // the main loop, then the CTAs meet.
    const int sub = lane >> 3, c8 = lane & 7, items = ((r1 - r0 + 3) / 4) * CHUNKS;
    const uint32_t base = smem_u32(tiles);
#pragma unroll 1
    for (int item = warp; item == warp || item < items; item += TILE_THREADS / 32) {
        const int group = item / CHUNKS, chunk = item % CHUNKS, r = r0 + group * 4 + sub;
        const int row = r < r1 ? m0 + r : g.M;                       // (g.M: a lane without a row)
        int ca, cb;
        chunk_halves<EPI, N_STEP>(chunk, g.d, ca, cb);
        const int col_a = n0 + ca + 4 * c8, col_b = n0 + cb + 4 * c8;
        const ColVals cv = load_cols<EPI>(g, col_a, col_b);
        const RowVals rv = load_row<EPI>(g, row, col_a, col_b);
        if (item == warp) {
            if (warp >= 4 && (warp & 3) * 32 < (SWAP ? BN : live)) {   // the partial tile into shared memory, over the ring: all its copies have landed and been read
                const int t = (warp & 3) * 32 + lane;                    // row of the tile; swapped: its column
                const uint32_t trow = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
                if (__all_sync(0xffffffffu, mbar_wait(&acc_full, 0, &abort_flag, g.wait_limit))) {
                    tc_fence_after();
                    if constexpr (SWAP) {
                        float *dst = reinterpret_cast<float *>(tiles);
#pragma unroll 1
                        for (int t0 = 0; t0 < live; t0 += 32) {
                            float hi[32], lo[32];
                            tmem_ld32(trow + t0, hi);
                            if (2 * g.a_rows <= 256) {
                                tmem_ld32(trow + g.a_rows + t0, lo);
                            } else {
#pragma unroll
                                for (int i = 0; i < 32; ++i) lo[i] = 0.f;
                            }
                            tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                if (t0 + i < live) dst[(t0 + i) * BN + ((((t >> 2) ^ (i & 7)) << 2) | (t & 3))] = hi[i] + lo[i];
                        }
                    } else {
                        float4 *dst = reinterpret_cast<float4 *>(tiles) + t * (BN / 4);
#pragma unroll 1
                        for (int c = 0; c < BN / 32; ++c) {
                            float v[32];
                            tmem_ld32(trow + c * 32, v);
                            tmem_ld_wait();
                            if (t < live) {
#pragma unroll
                                for (int q = 0; q < 8; ++q) dst[(c * 8 + q) ^ (t & 7)] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                            }
                        }
                    }
                    tc_fence_before();
                }
            }
            __syncwarp();
            if (S > 1) cluster_sync(); else __syncthreads();
            // of any CTA of the cluster: nothing is written
            const bool dead = S > 1 ? __any_sync(0xffffffffu, lane < S && cluster_ld1(cluster_addr(smem_u32(&abort_flag), lane)) != 0) : abort_flag != 0;
            if (dead || item >= items) {
                if (S > 1) cluster_arrive();
                break;
            }
        }
        const int rc = min(r, r1 - 1);
        const uint32_t off = base + rc * BN * 4, pa = off + ((ca / 4 + c8) ^ (rc & 7)) * 16, pb = off + ((cb / 4 + c8) ^ (rc & 7)) * 16;
        float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = va;
        if (S == 1) {
            va = *reinterpret_cast<const float4 *>(tiles + (pa - base));
            vb = *reinterpret_cast<const float4 *>(tiles + (pb - base));
        }
#pragma unroll 4
        for (int q = 0; q < S && S > 1; ++q) {        // in the order of K
            const float4 x = cluster_ld4(cluster_addr(pa, q)), y = cluster_ld4(cluster_addr(pb, q));
            va.x += x.x; va.y += x.y; va.z += x.z; va.w += x.w;
            vb.x += y.x; vb.y += y.y; vb.z += y.z; vb.w += y.w;
        }
        // Nobody leaves while its shared memory may still be read.  A warp arrives behind its last read, before it stores: an arrival that
        // releases stores to global memory waits for them (2.5 us).
        if (S > 1 && item + TILE_THREADS / 32 >= items) cluster_arrive();
        if (n0 + ca >= g.N) continue;        // a chunk past the matrix
        const float ss = finish_row<EPI>(g, row, col_a, col_b, va, vb, cv, rv, EPI == EPI_RESID ? 1.f : rs_sm[rc], 0);
        if (EPI == EPI_RESID && g.norm_w) store_row_ss(g, ss, row, n_tile * CHUNKS + chunk, lane);
    }
    if (warp == 1) {                         // (behind the barrier in the loop: the accumulator has been read)
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.tmem_cols) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) {    // (a CTA that has given up writes no partial tile over its ring)
        ring_land(full_bar, issued_sm, g.stages, g.extra_arrivals);
        atomicExch(g.error, 1);
    }
    if (S > 1) cluster_wait();
}

// ---- causal attention on tcgen05 ---------------------------------------------------------------------------------------------
// One CTA = 128 queries of one head (a query = a lane of tensor memory); keys in blocks of 128, dealt in turn to two groups of four
// softmax warps, which run half a block apart: while one group exponentiates, the tensor cores work for the other.  Per block j:
// S_j = Q K_j^T (tcgen05.mma, M 128, N 128, K = D; queries as two bf16 pieces) into the group's half of tensor memory;  a softmax
// thread owns a row: it reads its 128 scores twice (tcgen05.ld; once for the maximum, once for the exponentials), masks on diagonal
// blocks, and stores the probabilities as two bf16 pieces over the scores they came from (two keys per column; 32 scores become 16
// columns of hi and 16 of lo);  O += P_j V_j (M 128, N = D, K = 128 keys; P from tensor memory, V straight from its cache rows as an
// MN-major B operand), a sum of its own per group in tensor memory.  The exponentials are taken against a reference maximum that
// moves only when the row's maximum has grown by more than 2^8 (then the row of O and the row sum are rescaled once).  At the end
// the groups' sums meet in shared memory (those of the CTAs that share a query tile's key blocks in prefill_attention_merge_kernel).  The scores and P V are issued by two threads
// (warps 1 and 2), the K and V tiles have barriers of their own.
//   tensor memory: scores and probabilities [0, 128) and [128, 256), O [256, 256 + D) and [256 + D, 256 + 2 D)
//   shared memory: Q 2 x D/64 x 16 KB | 2 stages x (K D/64 x 16 KB, V D/64 x 16 KB)   (compressed cache: + landing areas)
// With one group of eight warps, two threads to a row, a block took 2.6 us, now 2.0: every block's chain of scores, maximum (exchanged between
// the two threads), exponentials and P V was walked with nothing beside it.  A prompt of 700 tokens behind 3000, 0.5B shape: 4067 -> 3635 us;
// 271 behind 1000, 1.5B: 4016 -> 3648; 2048, 1.5B: attention 43 -> 38 us a layer.
constexpr int AT_BM = 128, AT_BN = 128;
constexpr int AT_GROUPS = 2;
constexpr int AT_SPLIT_MAX = 16; // CTAs that share the key blocks of a query tile
constexpr int AT_CW = 8;       // compressed cache: warps that expand the codes (AT_BN / AT_CW rows of a tile each); with four of them, which
                               // fetched the scales behind the codes, 1000 tokens of the 3B shape took 12322 us instead of 12123
constexpr int AT_THREADS = 96 + 128 * AT_GROUPS;   // producer, two issuers, softmax warps

// B operand in MN-major form for P V: the V tile is D/64 blocks of [64 keys][64 d] (128-byte rows, 128-byte swizzle).  N (= d)
// runs along a row, K (= keys) across rows: groups of 8 keys are 1024 bytes apart (stride byte offset), the 64-column blocks
// `lbo` bytes apart (leading byte offset).
__device__ __forceinline__ uint64_t umma_desc_sw128_mn(uint32_t smem_addr, uint32_t lbo) {
    return static_cast<uint64_t>((smem_addr >> 4) & 0x3fffu) | (static_cast<uint64_t>((lbo >> 4) & 0x3fffu) << 16) | (64ull << 32) |
           (1ull << 46) | (2ull << 61);
}

template <int D> struct AttnCfg {
    static constexpr int KBLK = D / 64;                        // 64-column blocks of a row of q, k, v
    static constexpr int Q_BYTES = 2 * KBLK * AT_BM * 128;     // two pieces
    static constexpr int K_BYTES = KBLK * AT_BN * 128, V_BYTES = K_BYTES;
    static_assert(Q_BYTES == AT_BM * D * 4, "the rows of O pass through the place of Q, those of the second group through the first stage");
    static constexpr int SMEM = Q_BYTES + 2 * (K_BYTES + V_BYTES) + 1024;     // two stages of K and V
    // compressed cache: the 8-bit K tile has a landing area of its own, so that it can load while the scores of the blocks before still
    // read the operand tiles; a V tile lands in the first half of its operand tile's own place when a row of codes is as long as a
    // 128-byte operand row (D = 128: every row is then expanded in place; there is no room for more landing areas), D = 64 gets two
    static constexpr int RAW_BYTES = AT_BN * D;
    static constexpr int SMEM_Q8 = SMEM + (D == 128 ? 1 : 3) * RAW_BYTES;
    static constexpr int TMEM_COLS = 512;
};

template <int D, bool Q8>
__global__ void __launch_bounds__(AT_THREADS + (Q8 ? 32 * AT_CW : 0), Q8 ? 0 : 1) prefill_attention_tc_kernel(const __grid_constant__ CUtensorMap map_q_hi,
                                                                   const __grid_constant__ CUtensorMap map_q_lo,
                                                                   const __grid_constant__ CUtensorMap map_k,
                                                                   const __grid_constant__ CUtensorMap map_v, uint16_t *out, size_t plane,
                                                                   int T, int slot0, int nq, int group, int max_context,
                                                                   float scale_log2, uint32_t wait_limit, uint32_t extra_arrivals, int *error,
                                                                   const float *k_scale, const float *v_scale, float *part_o, float2 *part_ml) {
    // Q8: the cache holds 8-bit codes and a scale per row (k_scale, v_scale: this layer's [nkv][max_context]); map_k / map_v then
    // describe byte matrices; AT_CW more warps expand the codes to bf16 (exactly) into the operand layout, the softmax multiplies
    // the scores by the keys' scales and folds the values' scales into the probabilities.
    using C = AttnCfg<D>;
    extern __shared__ uint8_t at_tc_dyn[];
    __shared__ uint64_t kraw_full, kraw_empty, vraw_full[2];
    __shared__ __align__(16) float sc_k[Q8 ? 4 : 1][AT_BN], sc_v[Q8 ? 4 : 1][AT_BN];   // scales of the last four key blocks
    __shared__ uint64_t q_full, k_full[2], k_empty[2], v_full[2], v_empty[2], s_full[2], p_full[2][2], pv_done[2], all_done, drain_bar[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, issued_k, issued_v;  // key blocks whose K, V the producer has sent for
    __shared__ float2 row_ml[AT_GROUPS][AT_BM];     // reference maximum and sum of every row, at the end
    uint8_t *base = at_tc_dyn + ((1024u - (smem_u32(at_tc_dyn) & 1023u)) & 1023u);
    uint8_t *sq = base, *skv = sq + C::Q_BYTES, *sraw = skv + 2 * (C::K_BYTES + C::V_BYTES);   // sraw: landing areas of the codes (Q8)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // grid (heads, query tiles): CTAs start in linear order, so every head's longest tile (the last queries) starts first
    const int t0 = (gridDim.y - 1 - blockIdx.y) * AT_BM;
    const int h = blockIdx.x, hk = h / group;
    const int last_key = slot0 + min(t0 + AT_BM - 1, T - 1);
    // gridDim.z > 1 (a grid that would leave SMs idle): the key blocks of a query tile are shared out among gridDim.z CTAs;
    // each leaves its unnormalised rows of O, their reference maxima and sums in part_o / part_ml, prefill_attention_merge_kernel adds them
    const int nb_total = last_key / AT_BN + 1, splits = gridDim.z;
    const int j0 = static_cast<int>(blockIdx.z) * nb_total / splits;          // first key block of this CTA
    const int nb = (static_cast<int>(blockIdx.z) + 1) * nb_total / splits - j0;   // its key blocks (indices below are local)

    if (threadIdx.x == 0) {
        prefetch_map(&map_q_hi); prefetch_map(&map_q_lo); prefetch_map(&map_k); prefetch_map(&map_v);
        mbar_init(&q_full, 1 + extra_arrivals);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&k_full[i], Q8 ? AT_CW : 1); mbar_init(&k_empty[i], 1); mbar_init(&v_full[i], Q8 ? AT_CW : 1); mbar_init(&v_empty[i], 1);
            mbar_init(&vraw_full[i], 1); mbar_init(&s_full[i], 1); mbar_init(&pv_done[i], 1); mbar_init(&drain_bar[i], 1);
            mbar_init(&p_full[i][0], 4); mbar_init(&p_full[i][1], 4);
        }
        mbar_init(&kraw_full, 1); mbar_init(&kraw_empty, AT_CW); mbar_init(&all_done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(C::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_trigger();
    if (threadIdx.x == 0)                    // the cache rows are sent for to L2 (a hint: rows that are still being written are read later)
#pragma unroll 1
        for (int j = j0; j < j0 + min(nb, 4); ++j)
            for (int kb = 0; kb < (Q8 ? 1 : C::KBLK); ++kb) {
                prefetch_tile_l2(&map_k, kb * 64, hk * max_context + j * AT_BN);
                prefetch_tile_l2(&map_v, kb * 64, hk * max_context + j * AT_BN);
            }
    pdl_wait();   // set-up done; from here on the kernel reads what its predecessor wrote

    if (warp == 0 && lane == 0) {            // producer: the query tile once, then the K and V rows of every key block
        if (nb > 0) {
            mbar_expect_tx(&q_full, C::Q_BYTES);
            for (int kb = 0; kb < C::KBLK; ++kb) {
                tma_load_2d(sq + kb * AT_BM * 128, &map_q_hi, h * D + kb * 64, t0, &q_full);
                tma_load_2d(sq + (C::KBLK + kb) * AT_BM * 128, &map_q_lo, h * D + kb * 64, t0, &q_full);
            }
        }
        // K and V of a block have barriers of their own: the K tile is free again as soon as S_j is done, before the V tile, and the
        // next scores need only K.  Order of issue: K_0, then K_{j+1} before V_j, so that the wait for V's tile never holds the next
        // K tile back.  Block j uses stage j & 1.
        int nk = 0, nv = 0;
        auto load_k = [&](int j) {
            const int st = j & 1, y = hk * max_context + (j0 + j) * AT_BN;
            uint8_t *k = skv + st * (C::K_BYTES + C::V_BYTES);
            if constexpr (Q8) {
                if (j >= 1 && !mbar_wait(&kraw_empty, (j - 1) & 1, &abort_flag, wait_limit)) return false;
                mbar_expect_tx(&kraw_full, C::RAW_BYTES);
                tma_load_2d(sraw, &map_k, 0, y, &kraw_full);
            } else {
                if (j >= 2 && !mbar_wait(&k_empty[st], ((j >> 1) - 1) & 1, &abort_flag, wait_limit)) return false;
                mbar_expect_tx(&k_full[st], C::K_BYTES);
                for (int kb = 0; kb < C::KBLK; ++kb) tma_load_2d(k + kb * AT_BN * 128, &map_k, kb * 64, y, &k_full[st]);
            }
            nk = j + 1;
            return true;
        };
        auto load_v = [&](int j) {
            const int st = j & 1, y = hk * max_context + (j0 + j) * AT_BN;
            uint8_t *v = skv + st * (C::K_BYTES + C::V_BYTES) + C::K_BYTES;
            if (j >= 2 && !mbar_wait(&v_empty[st], ((j >> 1) - 1) & 1, &abort_flag, wait_limit)) return false;
            if constexpr (Q8) {
                mbar_expect_tx(&vraw_full[st], C::RAW_BYTES);
                tma_load_2d(D == 128 ? v : sraw + (1 + st) * C::RAW_BYTES, &map_v, 0, y, &vraw_full[st]);
            } else {
                mbar_expect_tx(&v_full[st], C::V_BYTES);
                for (int kb = 0; kb < C::KBLK; ++kb) tma_load_2d(v + kb * AT_BN * 128, &map_v, kb * 64, y, &v_full[st]);
            }
            nv = j + 1;
            return true;
        };
        bool ok = nb > 0 && load_k(0);
#pragma unroll 1
        for (int j = 0; j < nb && ok; ++j) {
            if (j + 1 < nb) ok = load_k(j + 1);
            if (ok) ok = load_v(j);
        }
        issued_k = nk;
        issued_v = nv;
    } else if (warp == 1 && lane == 0) {     // issuer of the scores: S_j = Q K_j^T, hi pieces then lo pieces
        // (two issuing threads, scores here and P V in warp 2: a tcgen05.mma takes about 40 ns to issue, and one thread issuing
        // both, with its six waits per block, was what bounded the kernel: 2.3 us per block)
        constexpr uint32_t idesc_s = umma_idesc_bf16(AT_BM, AT_BN);
        bool ok = nb == 0 || mbar_wait(&q_full, 0, &abort_flag, wait_limit);
#pragma unroll 1
        for (int j = 0; j < nb && ok; ++j) {
            const int g = j & 1, i = j >> 1;     // the group's i-th block
            ok = mbar_wait(&k_full[g], i & 1, &abort_flag, wait_limit);
            if (ok && i >= 1) ok = mbar_wait(&pv_done[g], (i - 1) & 1, &abort_flag, wait_limit);   // P_{j-2}, which lies over S_{j-2}, has been multiplied
            if (!ok) break;
            tc_fence_after();
            const uint32_t k = smem_u32(skv + g * (C::K_BYTES + C::V_BYTES)), acc = tmem + g * AT_BN;
#pragma unroll
            for (int piece = 0; piece < 2; ++piece)
#pragma unroll
                for (int kb = 0; kb < C::KBLK; ++kb) {
                    const uint64_t da = umma_desc_sw128(smem_u32(sq) + (piece * C::KBLK + kb) * AT_BM * 128);
                    const uint64_t db = umma_desc_sw128(k + kb * AT_BN * 128);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) umma_bf16(acc, da + 2 * kk, db + 2 * kk, idesc_s, (piece | kb | kk) != 0);
                }
            umma_commit(&s_full[g]);
            umma_commit(&k_empty[g]);        // the K rows are free when these have read them
        }
        if (!ok) {
            umma_commit(&drain_bar[0]);
            mbar_land(&drain_bar[0], 0);
        }
    } else if (warp == 2 && lane == 0) {     // issuer of O += P_j V_j, the block's two halves of 64 keys as they come
        constexpr uint32_t idesc_o = umma_idesc_bf16(AT_BM, D) | (1u << 16);   // B (= V) is MN-major
        bool ok = true;
#pragma unroll 1
        for (int j = 0; j < nb && ok; ++j) {
            const int g = j & 1, i = j >> 1;
            ok = mbar_wait(&v_full[g], i & 1, &abort_flag, wait_limit);
            const uint32_t v = smem_u32(skv + g * (C::K_BYTES + C::V_BYTES) + C::K_BYTES);
#pragma unroll
            for (int half = 0; half < 2 && ok; ++half) {
                ok = mbar_wait(&p_full[g][half], i & 1, &abort_flag, wait_limit);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int kg = 4 * half; kg < 4 * half + 4; ++kg)     // 16 keys: 8 columns of either piece of P, 2048 bytes of the V tile
#pragma unroll
                    for (int piece = 0; piece < 2; ++piece)
                        umma_bf16_ts(tmem + 2 * AT_BN + g * D, tmem + g * AT_BN + (kg >> 1) * 32 + piece * 16 + (kg & 1) * 8,
                                     umma_desc_sw128_mn(v + kg * 2048, AT_BN * 128), idesc_o, (i | kg | piece) != 0);
            }
            if (!ok) break;
            umma_commit(&pv_done[g]);
            umma_commit(&v_empty[g]);
        }
        if (ok) {
            umma_commit(&all_done);
        } else {
            umma_commit(&drain_bar[1]);
            mbar_land(&drain_bar[1], 0);
        }
    }
    else if (Q8 && warp >= AT_THREADS / 32) {   // compressed cache: expand the 8-bit tiles to bf16 operand tiles (AT_CW warps, AT_BN / AT_CW rows each)
        const int cw = warp - AT_THREADS / 32;
        constexpr int LPR = D / 16, RPS = 32 / LPR;       // lanes per row of codes (16 codes each), rows per step
        constexpr int ROWS = AT_BN / AT_CW;               // rows of a tile this warp expands
        auto warp_wait = [&](uint64_t *bar, int parity) {
            int r = 1;
            if (lane == 0) r = mbar_wait(bar, parity, &abort_flag, wait_limit) ? 1 : 0;
            return __shfl_sync(0xffffffffu, r, 0) != 0;
        };
        // 16 codes -> 16 bf16, exactly: byte b of (code + 128) under the exponent of 2^23 is the float 8388608 + code + 128
        auto expand = [&](uint4 c, uint4 &lo8, uint4 &hi8) {
            uint32_t w[4] = {c.x ^ 0x80808080u, c.y ^ 0x80808080u, c.z ^ 0x80808080u, c.w ^ 0x80808080u};
            uint32_t o[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float f0 = __uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7650)) - 8388736.f;
                const float f1 = __uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7651)) - 8388736.f;
                const float f2 = __uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7652)) - 8388736.f;
                const float f3 = __uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7653)) - 8388736.f;
                o[2 * i] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
                o[2 * i + 1] = __byte_perm(__float_as_uint(f2), __float_as_uint(f3), 0x7632);
            }
            lo8 = make_uint4(o[0], o[1], o[2], o[3]);
            hi8 = make_uint4(o[4], o[5], o[6], o[7]);
        };
        auto expand_tile = [&](uint8_t *tile, const uint8_t *raw) {
            // a lane takes 16 codes of a row per step; the warp loads the codes of ALL its rows before it stores anything (D = 128:
            // the operand rows overwrite the codes they came from), which also lets the loads overlap
            uint4 codes[ROWS / RPS];
#pragma unroll
            for (int step = 0; step < ROWS / RPS; ++step)
                codes[step] = *reinterpret_cast<const uint4 *>(raw + (cw * ROWS + step * RPS + lane / LPR) * D + (lane % LPR) * 16);
            __syncwarp();
#pragma unroll
            for (int step = 0; step < ROWS / RPS; ++step) {
                const int row = cw * ROWS + step * RPS + lane / LPR, c = lane % LPR;
                uint4 a, b;
                expand(codes[step], a, b);
                uint8_t *dst = tile + (c >> 2) * AT_BN * 128 + row * 128;
                *reinterpret_cast<uint4 *>(dst + (((2 * (c & 3)) ^ (row & 7)) << 4)) = a;
                *reinterpret_cast<uint4 *>(dst + (((2 * (c & 3) + 1) ^ (row & 7)) << 4)) = b;
            }
        };
        auto expand_k = [&](int j) {
            const int st = j & 1;
            // the scales of this block's keys (both kinds: they are in memory already), asked for before the codes are awaited: behind them
            // they put a trip to memory into every block
            static_assert(ROWS <= 32, "a lane per row");
            float ks = 0.f, vs = 0.f;
            if (lane < ROWS) {
                const size_t key = static_cast<size_t>(hk) * max_context + min((j0 + j) * AT_BN + cw * ROWS + lane, last_key);
                ks = k_scale[key];
                vs = v_scale[key];
            }
            if (!(warp_wait(&kraw_full, j & 1) && (j < 2 || warp_wait(&k_empty[st], ((j >> 1) - 1) & 1)))) return false;   // the codes are here, the operand tile is free
            expand_tile(skv + st * (C::K_BYTES + C::V_BYTES), sraw);
            __syncwarp();
            if (lane == 0) mbar_arrive(&kraw_empty);       // the next K tile may land
            if (lane < ROWS) {
                sc_k[j & 3][cw * ROWS + lane] = ks;
                sc_v[j & 3][cw * ROWS + lane] = vs;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&k_full[st]);
            return true;
        };
        bool ok = nb > 0 && expand_k(0);
#pragma unroll 1
        for (int j = 0; j < nb && ok; ++j) {              // like the producer: the next K tile before this block's V tile
            if (j + 1 < nb) ok = expand_k(j + 1);
            if (!ok) break;
            const int st = j & 1;
            ok = warp_wait(&vraw_full[st], (j >> 1) & 1);
            if (!ok) break;
            uint8_t *v = skv + st * (C::K_BYTES + C::V_BYTES) + C::K_BYTES;
            expand_tile(v, D == 128 ? v : sraw + (1 + st) * C::RAW_BYTES);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&v_full[st]);
        }
    }
    else if (warp >= 3) {                    // softmax: a thread per query row (= lane of tensor memory), the groups take blocks in turn
        const int quarter = warp & 3, g = (warp - 3) >> 2, row = quarter * 32 + lane;
        const uint32_t tlane = tmem + (static_cast<uint32_t>(quarter * 32) << 16), srow = tlane + g * AT_BN, orow = tlane + 2 * AT_BN + g * D;
        const int qi = slot0 + t0 + row;     // cache slot of this query: it sees the keys 0 .. qi
        // The output row accumulates in tensor memory over the blocks (P V with accumulation).  The exponentials are taken
        // against a reference maximum m_ref that moves only when the row's maximum has grown by more than 2^8 in the
        // exponent (or at the first block); then the row of O and the row sum are rescaled once.  In between the
        // probabilities may reach 2^8, which fp32 sums and the two bf16 pieces carry without loss.
        float m_ref = -1e30f, l_run = 0.f;   // (a row that sees none of its keys keeps a finite reference)
        bool ok = true;
        // one lane waits / arrives for its warp (an mbarrier operation per thread would cost more than the arithmetic)
        auto warp_wait = [&](uint64_t *bar, int parity) {
            int r = 1;
            if (lane == 0) r = mbar_wait(bar, parity, &abort_flag, wait_limit) ? 1 : 0;
            return __shfl_sync(0xffffffffu, r, 0) != 0;
        };
#pragma unroll 1
        for (int j = g; j < nb; j += AT_GROUPS) {
            const int i = j >> 1;
            ok = warp_wait(&s_full[g], i & 1);
            if (!ok) break;
            tc_fence_after();
            const int key0 = (j0 + j) * AT_BN;
            const bool diagonal = key0 + AT_BN - 1 > slot0 + t0;   // some query of the tile does not see the whole block
            auto receive = [&](int c, float *v) {       // 32 scores, scaled (Q8) and masked
                tmem_ld_ready(v);
                if constexpr (Q8) {                   // scores of codes -> scores: the keys' scales (16-byte shared-memory reads)
                    const float4 *sk = reinterpret_cast<const float4 *>(&sc_k[j & 3][c * 32]);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float4 f = sk[e];
                        v[4 * e] *= f.x; v[4 * e + 1] *= f.y; v[4 * e + 2] *= f.z; v[4 * e + 3] *= f.w;
                    }
                }
                if (diagonal) {
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (key0 + c * 32 + e > qi) v[e] = -INFINITY;
                }
            };
            // Both passes go over the chunks two by two, the next chunk's scores under way: eight chunks written out are more
            // instructions than the caches next to the schedulers hold, one at a time waits for every read.
            // (Compressed cache: one at a time all the same, its warps have registers for one.)
            constexpr bool PING = !Q8;
            float va[32], vb[PING ? 32 : 1];
            float mx = m_ref;
            auto fold = [&](const float *v) {
#pragma unroll
                for (int e = 0; e < 32; e += 4) mx = fmaxf(mx, fmaxf(fmaxf(v[e], v[e + 1]), fmaxf(v[e + 2], v[e + 3])));
            };
            tmem_ld32(srow, va);
#pragma unroll 1
            for (int c = 0; c < 4; c += PING ? 2 : 1) {      // pass 1: the maximum over the keys the query sees
                receive(c, va);
                if constexpr (PING) {
                    tmem_ld32(srow + (c + 1) * 32, vb);
                    fold(va);
                    receive(c + 1, vb);
                    tmem_ld32(srow + ((c + 2) & 3) * 32, va);     // (at the end: the first again)
                    fold(vb);
                } else {
                    fold(va);
                    tmem_ld32(srow + ((c + 1) & 3) * 32, va);
                }
            }
            if (i == 0) {
                m_ref = mx;
            } else if (__any_sync(0xffffffffu, (mx - m_ref) * scale_log2 > 8.f)) {
                // some row of this warp has outgrown its reference: every row moves its reference to its maximum and rescales its sum
                // and its row of O (the multiply of the group's block before is done: these scores lie where its probabilities lay)
                ok = warp_wait(&pv_done[g], (i - 1) & 1);
                if (!ok) break;
                tc_fence_after();
                const float f = fast_exp2((m_ref - mx) * scale_log2);
                l_run *= f;
#pragma unroll 1
                for (int c = 0; c < D / 32; ++c) {
                    float v[32];
                    tmem_ld32(orow + c * 32, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] *= f;
                    tmem_st32(orow + c * 32, v);
                }
                tmem_st_wait();
                m_ref = mx;
            }
            const float neg = -m_ref * scale_log2;
            float sum0 = 0.f, sum1 = 0.f;
            auto spend = [&](int c, const float *v) {     // probabilities as two bf16 pieces over the scores
                uint32_t phi[16], plo[16];        // two keys per word
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                    const float p0 = fast_exp2(fmaf(v[e], scale_log2, neg)), p1 = fast_exp2(fmaf(v[e + 1], scale_log2, neg));
                    sum0 += p0;
                    sum1 += p1;
                    if constexpr (Q8) {               // the values' scales ride on the probabilities
                        const float2 f = *reinterpret_cast<const float2 *>(&sc_v[j & 3][c * 32 + e]);
                        split2x2_trunc(p0 * f.x, p1 * f.y, phi[e / 2], plo[e / 2]);
                    } else {
                        split2x2_trunc(p0, p1, phi[e / 2], plo[e / 2]);
                    }
                }
                // P as the A operand in tensor memory: lane = query row, a column holds two consecutive keys (bf16)
                tmem_st16(srow + c * 32, reinterpret_cast<const float *>(phi));
                tmem_st16(srow + c * 32 + 16, reinterpret_cast<const float *>(plo));
            };
#pragma unroll 1
            for (int c = 0; c < 4; c += PING ? 2 : 1) {      // pass 2
                receive(c, va);
                if constexpr (PING) {
                    tmem_ld32(srow + (c + 1) * 32, vb);
                    spend(c, va);
                    receive(c + 1, vb);
                    if (c == 0) tmem_ld32(srow + 64, va);
                    spend(c + 1, vb);
                } else {
                    spend(c, va);
                    if (c < 3) tmem_ld32(srow + (c + 1) * 32, va);
                    if ((c & 1) == 0) continue;
                }
                tmem_st_wait();                   // a half is complete
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&p_full[g][c >> 1]);
            }
            l_run += sum0 + sum1;
        }
        if (ok && nb > 0) ok = warp_wait(&all_done, 0);   // the last multiply: Q, K and V have been read for the last time
        if (ok) {
            // the unnormalised row over the query tile / the first stage: 16-byte pieces, their index xor the row
            tc_fence_after();
            float4 *dst = reinterpret_cast<float4 *>(sq + g * C::Q_BYTES) + row * (D / 4);
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
                float v[32];
                if (g < nb) {
                    tmem_ld32(orow + c * 32, v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = 0.f;
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) dst[(c * 8 + e) ^ (row & 7)] = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            }
            row_ml[g][row] = make_float2(m_ref, l_run);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (!abort_flag) {
        // O = sum O_g 2^((m_g - M) c), L = sum l_g 2^((m_g - M) c) over the two groups, M = max m_g; a warp per row, D / 32 columns per lane: O / L, or (one of
        // several CTAs) O, M and L
        constexpr int V = D / 32;
        const int live = min(AT_BM, T - t0);
#pragma unroll 1
        for (int r = warp; r < live; r += AT_THREADS / 32 + (Q8 ? AT_CW : 0)) {
            const float2 a = row_ml[0][r], b = row_ml[1][r];
            const float top = fmaxf(a.x, b.x), wa = fast_exp2((a.x - top) * scale_log2), wb = fast_exp2((b.x - top) * scale_log2), l = fmaf(a.y, wa, b.y * wb);
            const float *x = reinterpret_cast<const float *>(sq) + r * D + (((lane * V / 4) ^ (r & 7)) << 2) + lane * V % 4, *y = x + C::Q_BYTES / 4;
            float o[V];
#pragma unroll
            for (int i = 0; i < V; ++i) o[i] = fmaf(x[i], wa, y[i] * wb);
            const size_t i = static_cast<size_t>(t0 + r) * nq + h;
            if (splits > 1) {
                const size_t slot = static_cast<size_t>(blockIdx.z) * gridDim.y * AT_BM * nq + i;
                if (lane == 0) part_ml[slot] = make_float2(top, l);
#pragma unroll
                for (int e = 0; e < V; e += 2) *reinterpret_cast<float2 *>(part_o + slot * D + lane * V + e) = make_float2(o[e], o[e + 1]);
                continue;
            }
            const float inv = 1.f / l;
            uint16_t *dst = out + i * D + lane * V;
#pragma unroll
            for (int e = 0; e < V; e += 2) {
                uint32_t hi, lo;
                split2x2(o[e] * inv, o[e + 1] * inv, hi, lo);
                *reinterpret_cast<uint32_t *>(dst + e) = hi;
                *reinterpret_cast<uint32_t *>(dst + plane + e) = lo;
            }
        }
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(AttnCfg<D>::TMEM_COLS) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) {    // the copies in flight land before this thread leaves and the shared memory is released (see ring_land)
        if (nb > 0) {
            for (uint32_t e = 0; e < extra_arrivals; ++e) mbar_arrive(&q_full);
            mbar_land(&q_full, 0);
        }
        if constexpr (Q8) {
            if (issued_k > 0) mbar_land(&kraw_full, (issued_k - 1) & 1);
            ring_land(vraw_full, issued_v, 2, 0);
        } else {
            ring_land(k_full, issued_k, 2, 0);
            ring_land(v_full, issued_v, 2, 0);
        }
        atomicExch(error, 1);
    }
}

// Adds the partial rows of query tiles whose key blocks were shared out: for row t and head h, M = max m_p,
// O = sum O_p 2^((m_p - M) c), L = sum l_p 2^((m_p - M) c), out = O / L as two bf16 planes.  A warp per row, D / 32 columns per lane, all parts'
// loads under way together.  (A cluster's CTAs merging through distributed shared memory took 11 us where these 2.6 us and the stores
// do: code that runs once per CTA comes from memory line by line, and the clusters of a full CTA per SM wait for a free GPC.)
static_assert(AT_SPLIT_MAX <= 32, "a lane per part");
template <int D>
__global__ void __launch_bounds__(128) prefill_attention_merge_kernel(const float *part_o, const float2 *part_ml, int parts, int rows, uint16_t *out, size_t plane, int T,
                                                                      int nq, float scale_log2) {
    pdl_trigger();
    pdl_wait();
    constexpr int V = D / 32;
    const int lane = threadIdx.x & 31, i = blockIdx.x * 4 + (threadIdx.x >> 5);    // row and head: t * nq + h
    if (i >= T * nq) return;
    const size_t part = static_cast<size_t>(rows) * nq;      // partial rows of a part
    float2 ml = make_float2(-INFINITY, 0.f);
    if (lane < parts) ml = part_ml[lane * part + i];
    const float top = warp_max(ml.x), w = lane < parts ? fast_exp2((ml.x - top) * scale_log2) : 0.f, inv = 1.f / warp_sum(ml.y * w);
    float acc[V] = {};
#pragma unroll 8
    for (int p = 0; p < parts; ++p) {
        const float *src = part_o + (p * part + i) * D + lane * V;
        const float f = __shfl_sync(0xffffffffu, w, p);
#pragma unroll
        for (int e = 0; e < V; e += 2) {
            const float2 x = *reinterpret_cast<const float2 *>(src + e);
            acc[e] = fmaf(x.x, f, acc[e]);
            acc[e + 1] = fmaf(x.y, f, acc[e + 1]);
        }
    }
    uint16_t *dst = out + static_cast<size_t>(i) * D + lane * V;
#pragma unroll
    for (int e = 0; e < V; e += 2) {
        uint32_t hi, lo;
        split2x2(acc[e] * inv, acc[e + 1] * inv, hi, lo);
        *reinterpret_cast<uint32_t *>(dst + e) = hi;
        *reinterpret_cast<uint32_t *>(dst + plane + e) = lo;
    }
}

// Launch with the programmatic-stream-serialization attribute (see pdl_trigger / pdl_wait), in clusters of that many CTAs.  Long passes
// gain, too, where their kernels are short: 1423 tokens, 0.5B shape 4455 -> 4023 us, 2541 tokens 6075 -> 5838; 2048, 1.5B 11205 -> 11065; 4200,
// 7B, no difference.  (Launched before the tensor memory was allocated the successors cost long passes 1 - 3 %.)
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(int cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args &&...args) {
    return launch_cluster(1, kernel, grid, block, smem, stream, static_cast<KArgs>(args)...);
}

// Clusters of c CTAs, one CTA per SM, that run at once: a cluster stays within a GPC.  Of 148 SMs, what cudaOccupancyMaxActiveClusters answered on each of
// five B200s; a table, so that the plan and with it the order of the sums depend on the sizes and the SM count alone (on a GPU with other GPCs a plan
// may take a second round);
// one tile more than that is a second round (1.5B shape, 152 tokens: O and down as 24 clusters of six took 14 us a layer more than 12 of eight).
int clusters_at_once(int c, int num_sms) {
    constexpr int AT_148[PF_CLUSTER_MAX + 1] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
    return AT_148[c] * num_sms / 148;
}
// Ring and shared memory of a CTA of prefill_tile_kernel with kb k-blocks: `rows` of activations (as loaded), tiles of bn columns.  deep: one CTA per SM
// where the k-blocks are many.  The partial tile lies over the ring and may be the larger of the two (256 columns; 217 and more rows swapped).
struct TileRoom { int stages, smem; };
TileRoom tile_room(int rows, int bn, bool swap, int kb, bool deep) {
    const int a_bytes = rows * PF_BK * 2, stage = 2 * a_bytes + bn * PF_BK * 2;
    // the multiplies read 128 rows of the operand that has 128, from the start of either piece or (swapped) of the weights: room behind the
    // last stage for those that are not loaded
    const int reach = (swap ? 2 : 1) * a_bytes + PF_BM * PF_BK * 2, slack = reach > stage ? reach - stage : 0;
    int stages = (TILE_SMEM - 1024 - slack) / stage;
    if (kb > 2 * stages && deep) stages = (TILE_SMEM_DEEP - 1024 - slack) / stage;
    if (stages > TILE_STAGES_MAX) stages = TILE_STAGES_MAX;
    if (stages > kb) stages = kb;
    const int ring = stages * stage + slack, partial = rows * bn * 4;
    return {stages, 1024 + (ring > partial ? ring : partial)};
}
// Clusters of c that run at once in a contraction of kb k-blocks: where two of its CTAs fit an SM, any that are no more than the SMs.  (Taken for granted
// for tiles of 256 columns, 0.5B shape, 450 tokens, QKV and O ran as 20 clusters of seven in two rounds: 2719 us a prompt, 2334 as it is.)
int tiles_at_once(int c, int kb, int rows, int bn, bool swap, int num_sms) {
    const int one = clusters_at_once(c, num_sms), two = num_sms / c < 2 * one ? num_sms / c : 2 * one;
    return tile_room(rows, bn, swap, (kb + c - 1) / c, true).smem <= TILE_SMEM ? two : one;
}

// Rows of an activation tile that are loaded, up to 256 tokens: whole groups of 8, of 16 where the pieces are multiplied one after the other.
int swapped_rows(int M) { return M <= PF_BM ? (M + 7) & ~7 : (M + 15) & ~15; }

// ---- host side ---------------------------------------------------------------------------------------------------------------
// Map of a row-major bf16 [rows][K] matrix; a box is box_rows rows x 64 columns (one 128-byte swizzled row each); rows and
// columns outside the matrix read as zero.  (No multicast is used with these maps.)
bool encode_operand_map(CUtensorMap *m, const void *base, long long rows, int K, int box_rows = 128) {
    TensorMapEncodeFn enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
    const cuuint32_t box[2] = {PF_BK, static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int EPI, int COLUMNS, bool PAIR>
const char *launch_gemm_cfg(const CUtensorMap &ma, const CUtensorMap &ml, const CUtensorMap &mb, const GemmArgs &g, int units, int workers, cudaStream_t s) {
    using C = GemmCfg<COLUMNS, PAIR>;
    if (cudaFuncSetAttribute(prefill_gemm_kernel<EPI, COLUMNS, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess)
        return "cudaFuncSetAttribute failed";
    const int ctas = PAIR ? 2 : 1;
    launch_cluster(ctas, prefill_gemm_kernel<EPI, COLUMNS, PAIR>, dim3((units < workers ? units : workers) * ctas), dim3(192), C::SMEM, s, ma, ml, mb, g);
    return cudaGetLastError() == cudaSuccess ? nullptr : "prefill GEMM launch failed";
}

template <int EPI, int BN, bool SWAP>
const char *launch_tile(const CUtensorMap &ma, const CUtensorMap &ml, const CUtensorMap &mb, GemmArgs &g, int num_sms, cudaStream_t s) {
    const int n_step = EPI == EPI_SWIGLU ? BN / 2 : BN, tiles = ((g.N + n_step - 1) / n_step) * (SWAP ? 1 : (g.M + PF_BM - 1) / PF_BM);
    const int kb = ((g.K + PF_BK - 1) / PF_BK + g.cluster - 1) / g.cluster;      // of the CTA with the most
    const TileRoom room = tile_room(g.a_rows, BN, SWAP, kb, tiles * g.cluster <= num_sms);
    g.stages = room.stages;
    // swapped: the pieces' columns (side by side where they fit one multiply) are read 32 at a time
    const int cols = SWAP ? (2 * g.a_rows <= 256 ? g.a_rows : 0) + (g.a_rows + 31) / 32 * 32 : BN;
    for (g.tmem_cols = 32; g.tmem_cols < cols;) g.tmem_cols *= 2;
    if (cudaFuncSetAttribute(prefill_tile_kernel<EPI, BN, SWAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILE_SMEM_DEEP) != cudaSuccess)
        return "cudaFuncSetAttribute failed";
    launch_cluster(g.cluster, prefill_tile_kernel<EPI, BN, SWAP>, dim3(tiles * g.cluster), dim3(TILE_THREADS), static_cast<size_t>(room.smem), s, ma, ml, mb, g);
    return cudaGetLastError() == cudaSuccess ? nullptr : "prefill contraction launch failed";
}

template <int EPI>
const char *launch_gemm(const uint16_t *a, size_t a_plane, const void *w, long long w_rows, GemmArgs &g, int num_sms, cudaStream_t s) {
    CUtensorMap ma, ml, mb;
    const PrefillPlan plan = prefill_plan(EPI, g.d, g.M, g.N, g.K, num_sms);
    g.cluster = plan.cluster;
    g.splits = plan.splits;
    g.bn = plan.columns;
    g.a_rows = g.cluster && (g.M < PF_BM || plan.swap) ? swapped_rows(g.M) : PF_BM;
    const int b_rows = EPI == EPI_SWIGLU ? (plan.columns == 128 ? 64 : 128) : plan.pairs ? plan.columns / 2 : plan.columns < 128 ? plan.columns : 128;
    if (!encode_operand_map(&ma, a, g.M, g.K, g.a_rows) || !encode_operand_map(&ml, a + a_plane, g.M, g.K, g.a_rows) ||
        !encode_operand_map(&mb, w, w_rows, g.K, b_rows))
        return "cuTensorMapEncodeTiled failed";
    if (EPI == EPI_RESID) {       // whole tiles have (columns + 63) / 64 pieces each, the last what is left of the matrix
        const int whole = (g.N - 1) / g.bn;
        g.ss_pieces = whole * ((g.bn + 63) / 64) + (g.N - whole * g.bn + 63) / 64;
    }
    if constexpr (EPI != EPI_LOGITS)
        if (g.cluster) {
            if constexpr (EPI != EPI_SWIGLU) {
                if (plan.columns == 256) return launch_tile<EPI, 256, false>(ma, ml, mb, g, num_sms, s);
                if (plan.columns == 64) return plan.swap ? launch_tile<EPI, 64, true>(ma, ml, mb, g, num_sms, s) : launch_tile<EPI, 64, false>(ma, ml, mb, g, num_sms, s);
            }
            return plan.swap ? launch_tile<EPI, 128, true>(ma, ml, mb, g, num_sms, s) : launch_tile<EPI, 128, false>(ma, ml, mb, g, num_sms, s);
        }
    const int m_tiles = (g.M + PF_BM - 1) / PF_BM;
    if constexpr (EPI != EPI_SWIGLU)
        if (plan.columns == 128) return launch_gemm_cfg<EPI, 128, false>(ma, ml, mb, g, m_tiles * ((g.N + 127) / 128) * g.splits, num_sms, s);
    const int n_step = EPI == EPI_SWIGLU ? 128 : g.bn, units = ((g.N + n_step - 1) / n_step) * g.splits;
    if constexpr (EPI != EPI_LOGITS)
        if (plan.pairs) return launch_gemm_cfg<EPI, 256, true>(ma, ml, mb, g, (m_tiles + 1) / 2 * units, num_sms / 2, s);
    return launch_gemm_cfg<EPI, 256, false>(ma, ml, mb, g, m_tiles * units, num_sms, s);
}

// Map of a byte matrix [rows][row_bytes] (the codes of a compressed cache); a box is box_rows whole rows, unswizzled.
bool encode_bytes_map(CUtensorMap *m, const void *base, long long rows, int row_bytes, int box_rows) {
    TensorMapEncodeFn enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(row_bytes), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(row_bytes)};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(row_bytes), static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// kc / vc: this layer's cache, bf16 rows or (k_scale != nullptr) rows of 8-bit codes with their scales.
// The key blocks of a query tile may be shared out (prefill_attention_parts); the partial rows are then merged (part_o / part_ml: room for num_sms tiles
// of 128 rows).
template <int D>
const char *launch_attention_tc(const uint16_t *q, const void *kc, const void *vc, const float *k_scale, const float *v_scale, uint16_t *out,
                                size_t plane, int T, int slot0, int nq, int nkv, int max_context, uint32_t wait_limit, uint32_t extra_arrivals, int *error,
                                float *part_o, float2 *part_ml, int num_sms, cudaStream_t s, int *launches) {
    const long long kv_rows = static_cast<long long>(nkv) * max_context;
    const bool q8 = k_scale != nullptr;
    CUtensorMap mqh, mql, mk, mv;
    if (!encode_operand_map(&mqh, q, T, nq * D) || !encode_operand_map(&mql, q + plane, T, nq * D)) return "cuTensorMapEncodeTiled failed";
    if (q8 ? (!encode_bytes_map(&mk, kc, kv_rows, D, AT_BN) || !encode_bytes_map(&mv, vc, kv_rows, D, AT_BN))
           : (!encode_operand_map(&mk, kc, kv_rows, D, AT_BN) || !encode_operand_map(&mv, vc, kv_rows, D, AT_BN)))
        return "cuTensorMapEncodeTiled failed";
    const float scale_log2 = static_cast<float>(1.4426950408889634 / sqrt(static_cast<double>(D)));
    const int tiles = (T + AT_BM - 1) / AT_BM, splits = prefill_attention_parts(T, slot0, nq, num_sms);
    const dim3 grid(nq, tiles, splits);
    if (q8) {
        if (cudaFuncSetAttribute(prefill_attention_tc_kernel<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<D>::SMEM_Q8) != cudaSuccess)
            return "cudaFuncSetAttribute failed";
        launch_pdl(prefill_attention_tc_kernel<D, true>, grid, dim3(AT_THREADS + 32 * AT_CW), AttnCfg<D>::SMEM_Q8, s, mqh, mql, mk, mv, out, plane, T,
                   slot0, nq, nq / nkv, max_context, scale_log2, wait_limit, extra_arrivals, error, k_scale, v_scale, part_o, part_ml);
    } else {
        if (cudaFuncSetAttribute(prefill_attention_tc_kernel<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<D>::SMEM) != cudaSuccess)
            return "cudaFuncSetAttribute failed";
        launch_pdl(prefill_attention_tc_kernel<D, false>, grid, dim3(AT_THREADS), AttnCfg<D>::SMEM, s, mqh, mql, mk, mv, out, plane, T, slot0, nq,
                   nq / nkv, max_context, scale_log2, wait_limit, extra_arrivals, error, static_cast<const float *>(nullptr), static_cast<const float *>(nullptr),
                   part_o, part_ml);
    }
    if (splits > 1)
        launch_pdl(prefill_attention_merge_kernel<D>, dim3((T * nq + 3) / 4), dim3(128), 0, s, static_cast<const float *>(part_o), static_cast<const float2 *>(part_ml),
                   splits, tiles * AT_BM, out, plane, T, nq, scale_log2);
    *launches += splits > 1 ? 2 : 1;
    return cudaGetLastError() == cudaSuccess ? nullptr : "prefill attention launch failed";
}

}  // namespace

// Few query tiles behind a long cache (a short suffix behind a prefix, a verified block) would run on few CTAs, each walking the whole cache: the key
// blocks are then shared out among as many CTAs as fit the SMs once.  Two blocks cost a CTA about 3.5 us (one for either group), the merge about
// as much.
int prefill_attention_parts(int T, int slot0, int nq, int num_sms) {
    const int blocks = (slot0 + T - 1) / AT_BN + 1, tiles = (T + AT_BM - 1) / AT_BM;
    int parts = 1;
    for (int c = 2, best = (blocks + 1) / 2; c <= AT_SPLIT_MAX && c * nq * tiles <= num_sms; ++c) {
        const int cost = ((blocks + c - 1) / c + 1) / 2 + 1;
        if (cost < best) { parts = c; best = cost; }
    }
    return parts;
}

// What a contraction is launched as (host logic, depends on the sizes and the SM count alone).
PrefillPlan prefill_plan(int epilogue, int head_dim, int M, int N, int K, int num_sms) {
    const int m_tiles = (M + PF_BM - 1) / PF_BM, kb = (K + PF_BK - 1) / PF_BK;
    auto rounds = [](int units, int n) { return (units + n - 1) / n; };
    auto tiles_of = [&](int step) { return m_tiles * ((N + step - 1) / step); };      // step: output columns a tile covers
    // What the persistent kernel would take with single CTAs: the rounds over the SMs times the cost of a unit; a tile of 256 columns does twice the
    // work of one of 128 for 1.33 x the operand traffic (1.6), a K split divides a unit's cost and adds a little for the partial sums (5 %).
    // Only the contractions that add to the residual stream split; a split keeps at least 12 k-blocks per unit and is considered only when the
    // unsplit tiles do not fill the SMs once (with more tiles the partial-sum traffic costs more than the better balance gains: 7B shape,
    // 2048 tokens, 48.0 -> 50.7 ms).  Gate/up: 128 gate columns and their 128 up columns.
    PrefillPlan p{256, 1, 0, false, false};
    if (epilogue != EPI_SWIGLU) {
        double best = 1e30;
        for (int columns = 128; columns <= 256; columns *= 2)
            for (int sp = 1; sp <= (epilogue == EPI_RESID ? (m_tiles == 1 ? PF_SPLIT_MAX : 4) : 1); ++sp) {
                if (sp > 1 && (kb / sp < 12 || tiles_of(columns) > num_sms)) break;
                const double t = rounds(tiles_of(columns) * sp, num_sms) * (columns == 256 ? 1.6 : 1.0) / sp * (sp > 1 ? 1.05 : 1.0);
                if (t < best - 1e-9) { best = t; p.columns = columns; p.splits = sp; }
            }
    }
    if (epilogue == EPI_LOGITS) return p;
    // Columns of the smallest tiles that clusters are made of: 64 (a QKV tile is whole heads; gate/up: 64 + 64) where those fit the SMs in one round
    // with the K split above, 128 where it has no use for more; else (0) the tiles are too many.
    int base = 0;
    if ((epilogue != EPI_QKV || head_dim == 64) && tiles_of(64) * p.splits <= num_sms) {
        base = epilogue == EPI_SWIGLU ? 128 : 64;
    } else if (p.columns == 128) {
        if (tiles_of(128) > num_sms) return p;
        base = 128;
    }
    // 129 to 256 tokens: the tokens as the columns of one row of tiles (gate/up: 64 + 64 columns), if these fit the SMs once and no other tiles that do
    // are cheaper.
    PrefillPlan wide_swap{128, 1, 0, false, true};
    int wide_swap_cost = 1 << 30;
    if (m_tiles == 2) {
        const int steps = (N + (epilogue == EPI_SWIGLU ? 63 : 127)) / (epilogue == EPI_SWIGLU ? 64 : 128), block = 4 * swapped_rows(M) + 2 * 128;
        for (int c = 1; c <= PF_CLUSTER_MAX && c <= kb && steps <= tiles_at_once(c, kb, swapped_rows(M), 128, true, num_sms); ++c) {
            const int cost = (kb + c - 1) / c * block + (c > 1 ? 2000 : 0);
            if (cost < wide_swap_cost) { wide_swap.cluster = c; wide_swap_cost = cost; }
        }
    }
    // Clusters where the tiles fit the SMs in one round.  A k-block costs a CTA what its operands take at 64 bytes per cycle, or its multiplies:
    // 4 cycles per column over 128 rows, or (swapped, the weights are the rows) 4 per token; sharing a tile's K costs the exchange of the
    // partial tiles, about 2000 cycles.  Tiles of 256 columns halve the traffic of several row tiles' activations.
    if (base) {
        const int rows = M < PF_BM ? (M + 7) & ~7 : PF_BM;
        int best = 1 << 30;
        for (int bn = base; bn <= (epilogue == EPI_SWIGLU || m_tiles == 1 ? base : 256); bn *= 2) {
            const int tiles = tiles_of(epilogue == EPI_SWIGLU ? bn / 2 : bn);
            const bool swap = rows < bn && bn <= 128 && rows < PF_BM;
            for (int c = 1; c <= PF_CLUSTER_MAX && c <= kb && tiles <= tiles_at_once(c, kb, rows, bn, swap, num_sms); ++c) {
                const int multiplies = 4 * (swap ? (rows > 32 ? rows : 32) : bn), operands = 4 * rows + 2 * bn;
                const int cost = (kb + c - 1) / c * (multiplies > operands ? multiplies : operands) + (c > 1 ? 2000 : 0);
                if (cost < best) { best = cost; p.columns = bn; p.cluster = c; p.swap = swap; }
            }
        }
        p.splits = 1;
        return wide_swap_cost < best ? wide_swap : p;
    }
    if (wide_swap.cluster) return wide_swap;
    // Gate/up of one row tile with more tiles than SMs: 64 + 64 columns, two CTAs per SM.  A pass over so many weights is bound by what an SM
    // asks for from memory at a time, and the persistent kernel's stages of 64 KB are half activations (64 tokens, 7B shape: 63 us for 271 MB;
    // the prompt 4355 -> 4185 us so).
    if (epilogue == EPI_SWIGLU && m_tiles == 1 && (N + 63) / 64 <= 2 * num_sms) {
        const int rows = M < PF_BM ? (M + 7) & ~7 : PF_BM;
        return PrefillPlan{128, 1, 1, false, rows < PF_BM};
    }
    // Pairs of CTAs where they need no more rounds over the SMs (an odd number of row tiles leaves one CTA of a pair without work).
    const int workers = num_sms / 2, m_pairs = (m_tiles + 1) / 2, n_step = epilogue == EPI_SWIGLU ? 128 : 256;
    if (m_tiles < 2 || workers < 1) return p;
    p.pairs = rounds(m_pairs * ((N + n_step - 1) / n_step) * p.splits, workers) <= rounds(tiles_of(n_step) * p.splits, num_sms);
    // A contraction that adds to the residual stream takes the number of columns that fills its rounds best: a k-block costs a CTA 4 cycles
    // per column in the tensor cores, or what its operands (32 KB of activations, 64 bytes per column) take at 64 bytes per cycle; a K split costs its
    // partial sums a pass through memory and the norm kernel (about a tenth).  (4096 tokens, 7B shape: 160 columns, 4.97 rounds, against 3.03
    // rounds of 256: O 212 -> 202 us, down 930 -> 894, at the power limit.)
    if (epilogue == EPI_RESID) {
        double best = p.pairs ? rounds(m_pairs * ((N + 255) / 256) * p.splits, workers) * 1024. / p.splits : rounds(tiles_of(256) * p.splits, num_sms) * 1075. / p.splits;
        if (p.splits > 1) best *= 1.05 * 1.1;
        for (int bn = 144; bn <= 256; bn += 16) {        // (128 columns are single CTAs' tiles, see launch_gemm)
            const double cost = rounds(m_pairs * ((N + bn - 1) / bn), workers) * static_cast<double>(4 * bn > 512 + bn ? 4 * bn : 512 + bn);
            if (cost < best - 1e-9) { best = cost; p.columns = bn; p.splits = 1; p.pairs = true; }
        }
    }
    return p;
}

size_t prefill_buffer_bytes(const edgefm_shape &sh, int chunk) {
    const size_t c = static_cast<size_t>(chunk), qd = static_cast<size_t>(sh.n_q_heads) * sh.head_dim;
    return c * sh.hidden * 4 * (1 + PF_SPLIT_MAX) + c * sh.hidden * 4 + c * PF_SS_PIECES(sh.hidden) * 4 + 2 * c * qd * 4 + c * sh.ffn * 4 + c * (sh.head_dim / 2) * 8 + c * 4 + 256;
}

cudaError_t prefill_alloc(PrefillBuffers *b, const edgefm_shape &sh, int chunk, bool kv8, int num_sms) {
    const size_t c = static_cast<size_t>(chunk), qd = static_cast<size_t>(sh.n_q_heads) * sh.head_dim;
    cudaError_t e;
    if ((e = cudaMalloc(&b->resid, c * sh.hidden * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->xn, c * sh.hidden * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->ss, c * PF_SS_PIECES(sh.hidden) * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->part, c * sh.hidden * 4 * PF_SPLIT_MAX)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->q, c * qd * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->attn, c * qd * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->act, c * sh.ffn * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->rope, c * (sh.head_dim / 2) * sizeof(float2))) != cudaSuccess) return e;
    if (kv8 && (e = cudaMalloc(&b->kv_stage, 2 * c * sh.n_kv_heads * sh.head_dim * sizeof(float))) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->tokens, c * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->error, 4)) != cudaSuccess) return e;
    b->logits_rows = sh.vocab;
    if ((e = cudaMalloc(&b->logits, static_cast<size_t>(PF_VERIFY_MAX) * sh.vocab * 4)) != cudaSuccess) return e;
    const size_t part_rows = static_cast<size_t>(num_sms) * AT_BM;
    if ((e = cudaMalloc(&b->att_o, part_rows * sh.head_dim * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->att_ml, part_rows * sizeof(float2))) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->head_val, PF_HEAD_GRID_MAX * PF_VERIFY_MAX * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->head_idx, PF_HEAD_GRID_MAX * PF_VERIFY_MAX * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->head_ticket, 4)) != cudaSuccess) return e;
    if ((e = cudaMemset(b->head_ticket, 0, 4)) != cudaSuccess) return e;
    if ((e = cudaMemset(b->error, 0, 4)) != cudaSuccess) return e;
    b->chunk = chunk;
    return cudaSuccess;
}

void prefill_free(PrefillBuffers *b) {
    cudaFree(b->resid); cudaFree(b->xn); cudaFree(b->part); cudaFree(b->ss); cudaFree(b->kv_stage); cudaFree(b->q); cudaFree(b->attn); cudaFree(b->act); cudaFree(b->rope);
    cudaFree(b->tokens); cudaFree(b->error); cudaFree(b->logits); cudaFree(b->att_o); cudaFree(b->att_ml); cudaFree(b->head_val); cudaFree(b->head_idx); cudaFree(b->head_ticket);
    *b = PrefillBuffers{};
}

const char *prefill_run(const PrefillModel &m, PrefillBuffers *b, const int32_t *tokens, int n, int slot0, int position, bool whole_last_layer,
                        cudaStream_t s, int *launches) {
    const edgefm_shape &sh = m.shape;
    const int H = sh.hidden, F = sh.ffn, d = sh.head_dim, nq = sh.n_q_heads, nkv = sh.n_kv_heads, qd = nq * d;
    const int n_qkv = (nq + 2 * nkv) * d;
    const long long head_stride = static_cast<long long>(m.max_context) * d;
    const size_t cap = static_cast<size_t>(b->chunk), x_plane = cap * H, q_plane = cap * qd, f_plane = cap * F;   // hi / lo planes
    int count = 0;
    if (cudaMemcpyAsync(b->tokens, tokens, static_cast<size_t>(n) * 4, cudaMemcpyHostToDevice, s) != cudaSuccess) return "token upload failed";
    // The first kernel of a pass is launched the plain way: it starts when everything enqueued before is complete, and so does, whatever overlaps
    // below, every kernel of the pass.  The contractions read weights before they wait for their predecessors; what an earlier kernel wrote
    // (weights a caller has changed, the rows of a vocabulary subset) is there by then.
    prefill_rope_kernel<<<dim3((n * (d / 2) + 255) / 256), dim3(256), 0, s>>>(b->rope, n, d / 2, position, static_cast<double>(sh.rope_theta));
    const int norm_grid = n;
    launch_pdl(prefill_norm_kernel, dim3(norm_grid), dim3(128), 0, s, b->resid, b->xn, x_plane, static_cast<const uint16_t *>(m.layers[0].input_norm),
                                                  static_cast<const uint16_t *>(m.embed), b->tokens, n, H, sh.rms_eps, m.state,
                                                  slot0 + n, position + n, nullptr, 0, 0);
    count += 2;
    int pieces = 0;
    bool raw = false;    // xn holds x * w of the residual stream, its sums of squares in b->ss (else normalised rows)
    for (int l = 0; l < sh.n_layers; ++l) {
        const edgefm_layer_weights &w = m.layers[l];
        const bool kv8 = m.k_scale != nullptr;   // compressed cache: one byte per element and a scale per row
        const size_t layer_rows = static_cast<size_t>(l) * nkv * m.max_context;
        uint16_t *kc = m.k_cache + static_cast<size_t>(l) * nkv * head_stride, *vc = m.v_cache + static_cast<size_t>(l) * nkv * head_stride;
        signed char *kc8 = reinterpret_cast<signed char *>(m.k_cache) + layer_rows * d, *vc8 = reinterpret_cast<signed char *>(m.v_cache) + layer_rows * d;
        GemmArgs g{};
        g.M = n; g.error = b->error; g.wait_limit = b->wait_limit; g.extra_arrivals = b->extra_arrivals;
        g.N = n_qkv; g.K = H;
        // a contraction that reads xn scales its results by 1 / rms where the rows are not normalised; one that adds to the residual stream
        // prepares xn for the next, or leaves K-split partial sums to the norm kernel
        g.ss_stride = cap; g.ss_pieces = pieces; g.eps = sh.rms_eps;
        g.xw = b->xn; g.x_plane = x_plane; g.ss_out = b->ss;
        g.ss_in = raw ? b->ss : nullptr;
        g.bias = sh.qkv_bias ? static_cast<const uint16_t *>(w.bqkv) : nullptr;
        if (g.bias && (reinterpret_cast<uintptr_t>(g.bias) & 15u)) return "edgefm_prefill reads bqkv in 16-byte pieces: the vector must be 16-byte aligned";
        g.rope = b->rope; g.q_out = b->q; g.q_plane = q_plane;
        g.k_rows = kc + static_cast<size_t>(slot0) * d; g.v_rows = vc + static_cast<size_t>(slot0) * d;
        g.nq = nq; g.nkv = nkv; g.d = d; g.head_stride = head_stride;
        if (kv8) { g.k_stage = b->kv_stage; g.v_stage = b->kv_stage + cap * nkv * d; g.stage_stride = static_cast<long long>(cap) * d; }
        if (const char *e = launch_gemm<EPI_QKV>(b->xn, x_plane, w.wqkv, n_qkv, g, m.num_sms, s)) return e;
        ++count;
        if (kv8) {   // the new rows, compressed into their cache slots (attention reads them from there, like every other row)
            launch_pdl(prefill_quantize_rows_kernel, dim3((2 * nkv * n + 7) / 8), dim3(256), 0, s, g.k_stage, g.v_stage, g.stage_stride, kc8, vc8, m.k_scale + layer_rows,
                                                                              m.v_scale + layer_rows, nkv, n, d, m.max_context, slot0);
            ++count;
        }
        if (l == sh.n_layers - 1 && !whole_last_layer) break;   // the rest of the last layer feeds nothing that is kept
        const void *ka = kv8 ? static_cast<const void *>(kc8) : kc, *va = kv8 ? static_cast<const void *>(vc8) : vc;
        const float *ksc = kv8 ? m.k_scale + layer_rows : nullptr, *vsc = kv8 ? m.v_scale + layer_rows : nullptr;
        const char *e = d == 64 ? launch_attention_tc<64>(b->q, ka, va, ksc, vsc, b->attn, q_plane, n, slot0, nq, nkv, m.max_context, b->wait_limit, b->extra_arrivals, b->error, b->att_o, b->att_ml, m.num_sms, s, &count)
                                : launch_attention_tc<128>(b->q, ka, va, ksc, vsc, b->attn, q_plane, n, slot0, nq, nkv, m.max_context, b->wait_limit, b->extra_arrivals, b->error, b->att_o, b->att_ml, m.num_sms, s, &count);
        if (e) return e;      // (attention and its merge are counted where they are launched)
        g.N = H; g.K = qd; g.resid = b->resid; g.part = b->part; g.part_plane = x_plane;
        g.norm_w = static_cast<const uint16_t *>(w.post_norm);
        if ((e = launch_gemm<EPI_RESID>(b->attn, q_plane, w.wo, H, g, m.num_sms, s))) return e;
        if (g.splits > 1) {
            launch_pdl(prefill_norm_kernel, dim3(norm_grid), dim3(128), 0, s, b->resid, b->xn, x_plane, g.norm_w, nullptr, nullptr, n, H,
                       sh.rms_eps, nullptr, 0, 0, b->part, g.splits, x_plane);
            ++count;
        }
        g.ss_in = g.splits > 1 ? nullptr : b->ss;
        g.N = F; g.K = H; g.act = b->act; g.act_plane = f_plane;
        if ((e = launch_gemm<EPI_SWIGLU>(b->xn, x_plane, w.w_gate_up, 2LL * F, g, m.num_sms, s))) return e;
        g.N = H; g.K = F;
        // behind the last layer nothing is normalised here (the norm kernel runs for the partial sums alone)
        const bool last = l + 1 == sh.n_layers;
        g.norm_w = last ? nullptr : static_cast<const uint16_t *>(m.layers[l + 1].input_norm);
        if ((e = launch_gemm<EPI_RESID>(b->act, f_plane, w.w_down, H, g, m.num_sms, s))) return e;
        if (g.splits > 1) {
            launch_pdl(prefill_norm_kernel, dim3(norm_grid), dim3(128), 0, s, b->resid, b->xn, x_plane,
                       last ? static_cast<const uint16_t *>(w.input_norm) : g.norm_w, nullptr, nullptr, n, H, sh.rms_eps, nullptr, 0, 0, b->part, g.splits, x_plane);
            ++count;
        }
        raw = g.splits == 1;
        pieces = g.ss_pieces;
        count += 3;
    }
    if (cudaGetLastError() != cudaSuccess) return "prefill kernel launch failed";
    if (launches) *launches = count;
    return nullptr;
}

const char *prefill_head(const PrefillModel &m, PrefillBuffers *b, int row, const void *final_norm, const void *lm, const int *ids, int rows,
                         float *logits_out, int *next_token_out, int token, int pos, cudaStream_t s) {
    const int H = m.shape.hidden;
    int grid = HEAD_CTAS_PER_SM * m.num_sms;
    if (grid > PF_HEAD_GRID_MAX) grid = PF_HEAD_GRID_MAX;
    if (grid * 8 > rows) grid = (rows + 7) / 8;
    if (H * 4 > 40 * 1024 &&
        cudaFuncSetAttribute(prefill_head_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, H * 4) != cudaSuccess)
        return "cudaFuncSetAttribute failed";
    launch_pdl(prefill_head_kernel, dim3(grid), dim3(256), static_cast<size_t>(H) * 4, s, b->resid + static_cast<size_t>(row) * H, static_cast<const uint16_t *>(final_norm),
                                                                     static_cast<const uint16_t *>(lm), ids, rows, H, m.shape.rms_eps, logits_out,
                                                                     next_token_out, b->head_val, b->head_idx, b->head_ticket, m.state, token, pos);
    return cudaGetLastError() == cudaSuccess ? nullptr : "prefill output layer launch failed";
}

const char *prefill_verify_head(const PrefillModel &m, PrefillBuffers *b, int n, const void *final_norm, const void *lm, const int *ids, int rows,
                                float *logits_out, int *n_accepted_out, int *next_token_out, int slot0, int pos, cudaStream_t s, int *launches) {
    // final norm of the block's rows (two bf16 planes), the logits of all rows as ONE contraction over the output matrix on the
    // tensor cores (into the caller's buffer or the work buffer), then the greedy tokens and the acceptance rule
    const int H = m.shape.hidden;
    const size_t x_plane = static_cast<size_t>(b->chunk) * H;
    float *logits = logits_out ? logits_out : b->logits;
    if (!logits_out && rows > b->logits_rows) return "block verification: the work buffer for the logits is too small";
    launch_pdl(prefill_norm_kernel, dim3(n), dim3(128), 0, s, b->resid, b->xn, x_plane, static_cast<const uint16_t *>(final_norm),
               static_cast<const uint16_t *>(nullptr), static_cast<const int *>(nullptr), n, H, m.shape.rms_eps, static_cast<StepState *>(nullptr), 0, 0,
               static_cast<const float *>(nullptr), 0, static_cast<size_t>(0));
    GemmArgs g{};
    g.M = n; g.N = rows; g.K = H; g.error = b->error; g.wait_limit = b->wait_limit; g.extra_arrivals = b->extra_arrivals;
    g.resid = logits;
    if (const char *e = launch_gemm<EPI_LOGITS>(b->xn, x_plane, lm, rows, g, m.num_sms, s)) return e;
    int grid = m.num_sms;
    if (grid > PF_HEAD_GRID_MAX) grid = PF_HEAD_GRID_MAX;
    if (grid * 256 > rows) grid = (rows + 255) / 256;
    launch_pdl(prefill_verify_pick_kernel, dim3(grid), dim3(256), 0, s, static_cast<const float *>(logits), ids, rows, n, static_cast<const int *>(b->tokens),
               b->head_val, b->head_idx, b->head_ticket, m.state, slot0, pos, n_accepted_out, next_token_out);
    *launches += 3;
    return cudaGetLastError() == cudaSuccess ? nullptr : "block verification output layer launch failed";
}

}  // namespace edgefm
