// The weight stream of the decode-step kernel: the order of its chunks, the ring, the L2 look-ahead.
#pragma once
#include "step_prims.cuh"

namespace edgefm {
namespace step {

// Calls f(p0, b0, p1, b1, is_kv) for every chunk of the whole step in order, until f returns false.  (Running pointers, nothing
// recomputed per chunk: the feeding thread's instructions per chunk bound the stream of small chunks; with the addresses
// derived anew for every chunk, 64-bit divisions among them, the output layer streamed at 3.1 instead of 6.7 TB/s.)
template <bool Q8, typename F>
__device__ __forceinline__ void for_each_chunk(const Ctx &c, F f) {
    const Shared &sh = c.sh();
    const StepParams &p = c.p();
    const int half = 1 << p.half_shift;
#pragma unroll 1
    for (int layer = 0; layer <= p.n_layers; ++layer) {
#pragma unroll 1
        for (int op = layer == p.n_layers ? ST_LM : ST_QKV; op <= (layer == p.n_layers ? ST_LM : ST_DN); ++op) {
            if (op == ST_O && sh.share.any) {                   // the cache rows come between the QKV and the O rows
                constexpr int E = Q8 ? 1 : 2;
                const size_t at = ((static_cast<size_t>(layer) * p.nkv + sh.share.g) * p.max_context + sh.share.t0) * (p.D * E);
                const unsigned char *k = reinterpret_cast<const unsigned char *>(p.k_cache) + at, *v = reinterpret_cast<const unsigned char *>(p.v_cache) + at;
#pragma unroll 1
                for (int t = sh.share.t0; t < sh.share.t1; t += ST_KV_BLOCK) {
                    const unsigned bytes = static_cast<unsigned>(min(ST_KV_BLOCK, sh.share.t1 - t) * p.D * E);
                    if (!f(k, bytes, v, bytes, true)) return;
                    k += bytes;
                    v += bytes;
                }
            }
            const StepLayer *L = c.layer(layer);
            const unsigned char *w = reinterpret_cast<const unsigned char *>(op == ST_QKV ? L->wqkv : op == ST_O ? L->wo : op == ST_GU ? L->w_gate_up
                                                                             : op == ST_DN ? L->w_down : c.head().lm_head);
            const unsigned row_bytes = static_cast<unsigned>(p.cols[op].K) * 2u;
            const int u0 = sh.u0[op], u1 = sh.u1[op];
            const bool paired = op_paired(op);
            const int most = paired ? p.cols[op].rows_per_chunk >> 1 : p.cols[op].rows_per_chunk, per_batch = units_per_batch(op);
            const size_t partner = static_cast<size_t>(op == ST_QKV ? half : p.F) * row_bytes;
            w += static_cast<size_t>(op == ST_QKV ? (u0 >> p.half_shift) * p.D + (u0 & (half - 1)) : u0) * row_bytes;
#pragma unroll 1
            for (int u = u0; u < u1;) {
                int n = min(most, min(u1 - u, per_batch - ((u - u0) & (per_batch - 1))));   // chunks do not cross the batches in which the sums are finished
                if (op == ST_QKV) n = min(n, half - (u & (half - 1)));                      // rows of one head are contiguous, heads are not
                const unsigned bytes = static_cast<unsigned>(n) * row_bytes;
                if (!f(w, bytes, w + partner, paired ? bytes : 0u, false)) return;
                w += bytes;
                u += n;
                if (op == ST_QKV && (u & (half - 1)) == 0) w += partner;                    // past the partner rows of the head just finished
            }
        }
    }
}

// One thread fills the ring ...
template <bool Q8>
__device__ __forceinline__ void feed_ring(Ctx &c) {
    Shared &sh = c.sh();
    const StepParams &p = c.p();
    unsigned long long once, keep;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(once));    // weights are read once per step
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(keep));
    const unsigned ring = static_cast<unsigned>(p.ring_bytes), limit = p.spin_limit, ring_at = smem_u32(c.ring());
    unsigned issued = 0, freed = 0;              // chunks copied / released so far
    unsigned at = 0, tail = 0;                   // next offset; start of the oldest chunk still in use
    unsigned sent = 0;                           // 16-byte units copied so far
    bool ok = true;
    for_each_chunk<Q8>(c, [&](const unsigned char *p0, unsigned b0, const unsigned char *p1, unsigned b1, bool kv) {
        const unsigned bytes = b0 + b1, need = (bytes + 127u) & ~127u;
        // room: chunks lie one behind the other and are never cut; the oldest are waited for until this one fits
        for (;;) {
            if (issued == freed) { at = 0; tail = 0; break; }
            if (issued - freed < ST_BARS) {
                if (at >= tail) {
                    if (ring - at >= need) break;
                    if (tail > need) { at = 0; break; }
                } else if (tail - at > need) break;
            }
            if (!mbar_wait(&sh.empty[freed & (ST_BARS - 1)], (freed / ST_BARS) & 1u, c.abort(), limit)) { ok = false; return false; }
            ++freed;
            tail = freed == issued ? at : *reinterpret_cast<volatile unsigned *>(&sh.chunk_at[freed & (ST_BARS - 1)]);
        }
        const unsigned b = issued & (ST_BARS - 1);
        unsigned long long *bar = &sh.full[b];
        *reinterpret_cast<volatile unsigned *>(&sh.chunk_at[b]) = at;
        mbar_expect_tx(bar, bytes);
        const unsigned long long policy = kv ? keep : once;
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(ring_at + at),
                     "l"(p0), "r"(b0), "r"(smem_u32(bar)), "l"(policy)
                     : "memory");
        if (b1)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(ring_at + at + b0),
                         "l"(p1), "r"(b1), "r"(smem_u32(bar)), "l"(policy)
                         : "memory");
        at += need;
        ++issued;
        sent += bytes >> 4;
        *reinterpret_cast<volatile unsigned *>(&sh.sent) = sent;
        return true;
    });
    if (!ok) {               // giving up: the copies in flight must land before the CTA's shared memory is released
        int dummy = 0;
        for (unsigned k = issued > ST_BARS ? issued - ST_BARS : 0; k < issued; ++k)
            mbar_wait(&sh.full[k & (ST_BARS - 1)], (k / ST_BARS) & 1u, &dummy, limit);
    }
}
// ... another asks L2 for what comes after it, at most prefetch_bytes ahead: the ring alone holds too little to keep HBM busy
// through the exchanges, and a refill from L2 comes at more than twice the rate of HBM.
template <bool Q8>
__device__ __forceinline__ void feed_l2(Ctx &c) {
    Shared &sh = c.sh();
    const unsigned ahead = static_cast<unsigned>(c.p().prefetch_bytes) >> 4;
    if (ahead == 0) return;
    unsigned pos = 0;
    for_each_chunk<Q8>(c, [&](const unsigned char *p0, unsigned b0, const unsigned char *p1, unsigned b1, bool) {
        pos += (b0 + b1) >> 4;
        unsigned spins = 0;
        int lead;                                // (differences: the counters may wrap)
        while ((lead = static_cast<int>(pos - *reinterpret_cast<volatile unsigned *>(&sh.sent))) > static_cast<int>(ahead)) {
            if (*c.abort() || ++spins > (1u << 22)) return false;      // bounded; a hint not given costs only time
            __nanosleep(64);
        }
        if (lead <= 0) return true;              // the ring has it already
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p0), "r"(b0) : "memory");
        if (b1) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p1), "r"(b1) : "memory");
        return true;
    });
}

}  // namespace step
}  // namespace edgefm
