// Primitives of the decode-step kernel: barriers, bounded waits, packets.
#pragma once
#include "step_types.h"

// These headers are built twice.  ST_TIGHT: for shapes that leave the shared memory no room for the tables and the chunk list, or for chunks of
// the usual size.  (As run-time choices in the one kernel they cost every shape 1 - 4 %.)
#ifndef ST_TIGHT
#define ST_TIGHT 0
#endif
#if ST_TIGHT
#define ST_NS step_tight
#else
#define ST_NS step
#endif

namespace edgefm {
namespace ST_NS {

constexpr bool TIGHT = ST_TIGHT != 0;
constexpr int ROW_BITS = TIGHT ? ST_TIGHT_ROW_BITS : 16;     // of a unit table's entry: row | values << ROW_BITS | unit << (ROW_BITS + 2)
__device__ __forceinline__ int kv_positions(const StepParams &p, int D) { return TIGHT ? p.kv_block : kv_block(D); }   // cached positions per ring chunk

__device__ __forceinline__ unsigned smem_u32(const void *p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(unsigned long long *b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *b, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bookkeeping of a bounded wait: called after every unsuccessful poll, false = give up.
struct Spin {
    unsigned it = 0;
    unsigned long long t0 = 0;
    __device__ __forceinline__ bool again(volatile int *abort_flag, unsigned limit_ns) {
        if ((++it & 127u) == 0u) {
            if (*abort_flag) return false;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit_ns) { *abort_flag = 1; return false; }
        }
        return true;
    }
};
// The same for a warp whose lanes poll together: they leave together, too.  (Lanes that leave one by one stay apart for a while, and the
// shuffles behind the loop then cost microseconds: CTAs that had waited long were 3 - 4 us late at the next exchange.)
// -1: everything is there, 0: gave up, 1: poll again.
__device__ __forceinline__ int warp_again(Spin &sp, bool waiting, volatile int *abort_flag, unsigned limit_ns) {
    if (!__any_sync(0xffffffffu, waiting)) return -1;
    return __any_sync(0xffffffffu, !sp.again(abort_flag, limit_ns)) ? 0 : 1;
}
__device__ __forceinline__ bool mbar_wait(unsigned long long *b, unsigned parity, volatile int *abort_flag, unsigned limit_ns) {
    if (mbar_try_wait(b, parity)) return true;
    Spin sp;
    while (sp.again(abort_flag, limit_ns))
        if (mbar_try_wait(b, parity)) return true;
    return false;
}
// All consumer threads meet; true = every one of them came with ok (the decision is the same for all, so that nobody is left
// waiting at the next one).
__device__ __forceinline__ bool cta_vote(bool ok) {
    unsigned bad;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.eq.u32 q, %1, 0;\n\t"
        "barrier.cta.red.or.pred p, 1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(bad)
        : "r"(ok ? 1u : 0u), "n"(ST_NT)
        : "memory");
    return bad == 0;
}

// Packets.  Each 8-byte element of a vector access is written and read as a whole.
__device__ __forceinline__ unsigned long long packet(float v, unsigned tag) {
    return static_cast<unsigned long long>(tag) << 32 | __float_as_uint(v);
}
__device__ __forceinline__ float packet_value(unsigned long long p) { return __uint_as_float(static_cast<unsigned>(p)); }
__device__ __forceinline__ unsigned packet_tag(unsigned long long p) { return static_cast<unsigned>(p >> 32); }
__device__ __forceinline__ void put1(unsigned long long *at, float v, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(at), "l"(packet(v, tag)) : "memory");
}
__device__ __forceinline__ void put2(unsigned long long *at, float a, float b, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(at), "l"(packet(a, tag)), "l"(packet(b, tag)) : "memory");
}
// (Initialised where it is declared: a register that is only written under a predicate counts as live before it, in a persistent
// loop everywhere, and the kernel then spills around everything else.)
struct Two { unsigned long long a = 0ull, b = 0ull; };
__device__ __forceinline__ Two get2(const unsigned long long *at) {
    Two t;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(t.a), "=l"(t.b) : "l"(at) : "memory");
    return t;
}
struct Four { unsigned long long a = 0ull, b = 0ull, c = 0ull, d = 0ull; };
__device__ __forceinline__ Four get4(const unsigned long long *at) {
    Four t;
    asm volatile("ld.relaxed.gpu.global.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(t.a), "=l"(t.b), "=l"(t.c), "=l"(t.d) : "l"(at) : "memory");
    return t;
}
__device__ __forceinline__ bool both(const Two &t, unsigned tag) { return packet_tag(t.a) == tag && packet_tag(t.b) == tag; }

// Packets of pieces: three bf16 (value = their sum) and the low 16 bits of the tag.  A slot is rewritten with the next tag every layer
// (every token's, used or not), so 16 bits tell the contents apart.
__device__ __forceinline__ unsigned long long pieces_packet(float v, unsigned tag) {
    const uint16_t hi = f32_to_bf16_bits(v);
    v -= bf16_bits_to_f32(hi);           // exact: the remainder is what the next piece holds
    const uint16_t mid = f32_to_bf16_bits(v);
    const uint16_t lo = f32_to_bf16_bits(v - bf16_bits_to_f32(mid));
    return static_cast<unsigned long long>(hi | static_cast<unsigned>(mid) << 16) | static_cast<unsigned long long>(lo | tag << 16) << 32;
}
__device__ __forceinline__ bool pieces_tag(unsigned long long p, unsigned tag) { return static_cast<unsigned>(p >> 48) == (tag & 0xffffu); }
__device__ __forceinline__ void put_raw(unsigned long long *at, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(at), "l"(v) : "memory");
}
__device__ __forceinline__ void put_raw2(unsigned long long *at, unsigned long long a, unsigned long long b) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(at), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ unsigned long long get1(const unsigned long long *at) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(at) : "memory");
    return v;
}

__device__ __forceinline__ float exp2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sum8(const float *at) {
    const float4 a = *reinterpret_cast<const float4 *>(at), b = *reinterpret_cast<const float4 *>(at + 4);
    return ((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w));
}

// ---- shared memory ---------------------------------------------------------------------------------------------------
// Dynamic: Shared | ring | layer table, unit tables, residual rows | one area for the staged vector, the attention's scratch and the
// segments of the MLP activations (they follow one another; between the last reader of one and the first writer of the next
// lies a CTA-wide vote).
extern __shared__ __align__(128) unsigned char st_smem[];
template <int MT> struct Shared {
    unsigned long long full[ST_BARS], empty[ST_BARS];
    unsigned long long x_full[4], x_empty[4];              // staged vectors / segments of the MLP activations
    unsigned chunk_at[ST_BARS];                            // ring offset of the chunk behind every barrier
    float rope[MT][128];                                   // per token: cos | sin of its position
    float ss[MT];                                          // sums of squares (RMSNorm)
    alignas(16) float part[2][MT * st_batch(MT) * ST_NW];  // partial row sums [token][row][warp], two batches
    alignas(16) float merged[MT][128];                     // attention outputs this CTA owns (Ctx::merged)
    float best_v[ST_NW];
    int best_i[ST_NW];
    int u0[5], u1[5];                                      // this CTA's units of every operator
    int list[6];                                           // first entry of every operator in the chunk list
    unsigned tag0, odd;                                    // tag of layer 0; test hook: a bit no tag has
    int total_x, total_a;                                  // sizes of the unit tables
    int tokens[MT];
    int m, pos, n_old, n_chunks;                           // the call's tokens, first position, cache length; attention chunks per kv head and token
    unsigned sent;                                         // 16-byte units the feeding warp has asked for
    int abort;
};
template <int MT> __host__ __device__ constexpr int st_shared_bytes() { return (static_cast<int>(sizeof(Shared<MT>)) + 127) / 128 * 128; }

// What the device functions share: the parameter block (constant bank), the thread's place and the ring position; everything else
// stands in shared memory, so that little is carried in registers from one operator to the next.
template <int MT> struct Ctx {
    static constexpr int S = st_pieces(MT), NA = st_arrays(MT), RB = st_batch(MT);
    const StepParams &par;
    int tid, warp, lane, cta, ncta;
    unsigned chunk, xchunk;  // next ring chunk / staged vector to consume
    int act_slot;            // MLP activations: which of the segments in shared memory is next
    __device__ __forceinline__ explicit Ctx(const StepParams &p_)
        : par(p_), tid(static_cast<int>(threadIdx.x)), warp(tid >> 5), lane(tid & 31), cta(static_cast<int>(blockIdx.x)), ncta(static_cast<int>(gridDim.x)), chunk(0u), xchunk(0u), act_slot(0) {}
    __device__ __forceinline__ Shared<MT> &sh() const { return *reinterpret_cast<Shared<MT> *>(st_smem); }
    __device__ __forceinline__ const StepParams &p() const { return par; }
    __device__ __forceinline__ volatile int *abort() const { return &sh().abort; }
    __device__ __forceinline__ unsigned char *ring() const { return st_smem + st_shared_bytes<MT>(); }
    __device__ __forceinline__ unsigned char *tables() const { return ring() + p().ring_bytes; }
    __device__ __forceinline__ const StepLayer *layer(int l) const { return reinterpret_cast<const StepLayer *>(tables()) + l; }
    __device__ __forceinline__ const StepHead &head() const { return *reinterpret_cast<const StepHead *>(layer(p().n_layers)); }
    __device__ __forceinline__ unsigned *unit_table() const { return reinterpret_cast<unsigned *>(tables() + (p().n_layers + 1) * 64); }
    __device__ __forceinline__ uint4 *list() const { return reinterpret_cast<uint4 *>(tables() + p().list_at); }           // chunk list
    __device__ __forceinline__ float *resid() const { return reinterpret_cast<float *>(tables() + p().resid_at); }   // [token][this CTA's rows of the residual stream]
    __device__ __forceinline__ float *merged(int tok) const {      // attention outputs this CTA owns
        return TIGHT ? reinterpret_cast<float *>(tables() + p().merged_at) + tok * p().merged_len : sh().merged[tok];
    }
    __device__ __forceinline__ unsigned char *area() const { return tables() + p().table_bytes; }
};

template <int MT> __device__ __forceinline__ void stamp(const Ctx<MT> &c, int &idx) {
    const StepParams &p = c.p();
    if (p.prof && c.tid == 0) {
        if (idx < p.prof_stride) p.prof[static_cast<size_t>(c.cta) * p.prof_stride + idx] = global_ns();
        ++idx;
    }
}

// ---- ring: consumer side -----------------------------------------------------------------------------------------------
template <int MT> __device__ __forceinline__ bool chunk_wait(Ctx<MT> &c, const unsigned char *&at) {
    Shared<MT> &sh = c.sh();
    const unsigned b = c.chunk & (ST_BARS - 1), parity = (c.chunk / ST_BARS) & 1u;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[b], parity, c.abort(), c.p().spin_limit));
    at = c.ring() + *reinterpret_cast<volatile unsigned *>(&sh.chunk_at[b]);
    return ok;
}
template <int MT> __device__ __forceinline__ void chunk_release(Ctx<MT> &c) {
    __syncwarp();
    if (c.lane == 0) mbar_arrive(&c.sh().empty[c.chunk & (ST_BARS - 1)]);
    ++c.chunk;
}

__device__ __forceinline__ void store_u16(unsigned char *at, uint16_t v) { *reinterpret_cast<uint16_t *>(at) = v; }
// The pieces of value v to column `col` of token tok's arrays (`stride` bytes apart) at `base`.
template <int MT> __device__ __forceinline__ void store_pieces(unsigned char *base, int tok, int col, int stride, float v) {
    unsigned char *at = base + static_cast<size_t>(tok * Ctx<MT>::S) * stride + col * 2;
#pragma unroll
    for (int i = 0; i < Ctx<MT>::S; ++i) {
        const uint16_t b = f32_to_bf16_bits(v);
        store_u16(at, b);
        v -= bf16_bits_to_f32(b);        // exact: the remainder is what the next piece holds
        at += stride;
    }
}

template <int MT> __device__ __forceinline__ void store_packet(unsigned char *base, int tok, int col, int stride, unsigned long long v) {
    unsigned char *at = base + tok * Ctx<MT>::S * stride + col * 2;
#pragma unroll
    for (int i = 0; i < Ctx<MT>::S; ++i) store_u16(at + i * stride, static_cast<uint16_t>(v >> (16 * i)));
}
// Columns past K of the last 64-column block are multiplied by zero.
template <int MT> __device__ __forceinline__ void zero_tail(const Ctx<MT> &c, int K) {
    const int pad = (64 - (K & 63)) & 63, stride = st_array_bytes(K);
    for (int i = c.tid; i < pad * Ctx<MT>::NA; i += ST_NT) store_u16(c.area() + (i / pad) * stride + (K + i % pad) * 2, 0);
}

// ---- exchanges by arrival: every CTA has written its share of a vector to global memory ------------------------------------
// One thread arrives for the CTA.  (The thread that issues the copies puts the proxy fence between what it has acquired and the copies;
// a second one here, by every writer, cost each exchange 1 us.)
template <int MT> __device__ __forceinline__ bool arrive(const Ctx<MT> &c, bool ok) {
    ok = cta_vote(ok);
    if (ok && c.tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(c.p().arrivals) : "memory");
    return ok;
}
template <int MT> __device__ __forceinline__ bool x_wait(Ctx<MT> &c) {
    const unsigned b = c.xchunk & 3u;
    return __all_sync(0xffffffffu, mbar_wait(&c.sh().x_full[b], (c.xchunk >> 2) & 1u, c.abort(), c.p().spin_limit));
}
template <int MT> __device__ __forceinline__ void x_release(Ctx<MT> &c) {
    __syncwarp();
    if (c.lane == 0) mbar_arrive(&c.sh().x_empty[c.xchunk & 3u]);
    ++c.xchunk;
}

// ---- the order of the stream (the same arithmetic on the feeding and on the consuming side) --------------------------------
__host__ __device__ __forceinline__ int op_units(const StepParams &p, int op, int lm_rows) {
    switch (op) {
        case ST_QKV: return (p.nq + 2 * p.nkv) << p.half_shift;
        case ST_GU: return p.F;
        case ST_LM: return lm_rows;
        default: return p.H;
    }
}
__host__ __device__ __forceinline__ bool op_paired(int op) { return op == ST_QKV || op == ST_GU; }
// Units of the tile that starts at unit u of [.., u1).
__host__ __device__ __forceinline__ int tile_units(const StepParams &p, int op, int u, int u1) {
    int n = min(p.cols[op].tile, u1 - u);
    if (op == ST_QKV) n = min(n, (1 << p.half_shift) - (u & ((1 << p.half_shift) - 1)));   // rows of one head are contiguous, heads are not
    return n;
}
// Attention is dealt out by (token, kv head, chunk of the n_old cached positions); a CTA serves the shares cta, cta + ncta, ...
struct KvShare { int tok, g, chunk, t0, t1, tail; };
__device__ __forceinline__ int kv_chunks(const StepParams &p, int n, int m, int ncta) { return max(1, min(ncta / (p.nkv * m), (n + ST_MIN_CHUNK - 1) / ST_MIN_CHUNK)); }
__device__ __forceinline__ KvShare kv_share(const StepParams &p, int n, int n_chunks, int idx) {
    KvShare s;
    const int tg = idx / n_chunks;
    s.chunk = idx - tg * n_chunks;
    s.tok = tg / p.nkv;
    s.g = tg - s.tok * p.nkv;
    s.t0 = st_first(n, s.chunk, n_chunks);
    s.t1 = st_first(n, s.chunk + 1, n_chunks);
    s.tail = s.chunk == n_chunks - 1;
    return s;
}

}  // namespace ST_NS
}  // namespace edgefm
