// The whole decode step as ONE persistent cooperative kernel (one CTA per SM): every warp owns a slice of the COLUMNS.
//
// At batch 1 a step is a chain of matrix-vector products bound by the one pass over the weights, but cut by six exchanges per
// layer in which every SM needs what the others computed.  Two things decide its time: that the weight stream never stops,
// and what an exchange costs.
//
//   * Weights (step_feed.cuh).  A CTA owns a contiguous range of the rows of every operator, i.e. a contiguous range of memory.
//     One thread feeds a ring in shared memory with bulk copies (cp.async.bulk, 24 - 50 KB each) in the order of the whole step --
//     QKV rows, this CTA's K/V cache rows, O rows, gate/up rows, down rows, next layer, ..., output layer -- independent of the
//     computation; another asks L2 for what comes after the ring.  (A bulk copy costs its issuer the same few hundred cycles
//     whatever its size: measured from L2, 6 / 24 / 48 KB copies from one such loop reached 2.2 / 9 / 18 TB/s over the chip.)
//   * Products (step_products.cuh).  All 8 consumer warps work on every row; warp w multiplies columns [K w / 8, K (w + 1) / 8) with
//     its slice of the input vector, fp32.  bf16 weights become fp32 by a shift or a mask, products and sums are packed fp32
//     FMAs.  Row sums: shuffles over the lanes of a row (several rows folded at once), then the 8 partial sums of a row meet in
//     shared memory and one thread per output unit runs the fused epilogue (bias + RoPE + cache row, residual add, SwiGLU,
//     logits + argmax).
//   * Exchanges.  A value travels as an 8-byte packet {fp32 value, tag}; the tag names step and layer, so a reader polls the data
//     itself: one trip to L2 instead of store, fence, counter, poll, load.  Every CTA writes its values into a 128-byte line of
//     its own (packets of several writers in one line cost 0.3 - 1 us: the pollers' copies of the line are invalidated by every
//     write).  Measured, 148 CTAs, 1536 values everywhere: 1.3 us per round, against 1.7 us for a counter barrier and a read
//     (which leaves out the staging of the vector).  A buffer is rewritten one layer later; a CTA that writes it then has
//     read, in between, an exchange to which every CTA contributes only after reading the old contents.
//   * Attention (step_attention.cuh).  CTA (kv head, chunk) holds the chunk's K/V rows in its ring before the queries exist, serves
//     the whole GQA group from one read, and publishes unnormalised partial results; the owner of an output pair merges them
//     (one warp per pair, lanes over chunks) and publishes the finished vector.  The row this step appends travels as packets too.
//
// Every wait is bounded: on expiry the CTA records status 6, all its warps leave at the next CTA-wide vote, the feeding thread
// waits (bounded) for its copies in flight.
#include "step_attention.cuh"
#include "step_feed.cuh"
#include "step_products.cuh"

namespace edgefm {
namespace step {

// The epilogue of output unit j (its row sum, or the sums of its two rows) of an operator.
template <int D, bool Q8>
__device__ __forceinline__ void finish_unit(const Ctx &c, int op, int layer, int j, int u0, float lo, float hi, float add_lo, float add_hi, float &best_v,
                                            int &best_i) {
    const Shared &sh = c.sh();
    const StepParams &p = c.p();
    constexpr int half = D / 2;
    const unsigned tag = sh.tag0 + static_cast<unsigned>(layer);
    if (op != ST_O && op != ST_DN) {       // the deferred RMSNorm factor
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < ST_NW; ++w) tot += sh.ss[w];
        const float r = rsqrtf(tot / static_cast<float>(p.H) + p.eps);
        lo *= r;
        hi *= r;
    }
    if (op == ST_QKV) {
        const int head = j >> p.half_shift, i = j & (half - 1);
        lo += add_lo;
        hi += add_hi;
        if (head < p.nq + p.nkv) {
            const float cs = sh.rope[i], sn = sh.rope[half + i];
            const float a = lo * cs - hi * sn, b = hi * cs + lo * sn;
            lo = a;
            hi = b;
        }
        put2(p.q_ll + static_cast<size_t>(c.cta) * p.q_line + 2 * (j - u0), lo, hi, tag);
        if (!Q8 && head >= p.nq) {
            const bool is_v = head >= p.nq + p.nkv;
            const int g = head - p.nq - (is_v ? p.nkv : 0);
            uint16_t *d = (is_v ? p.v_cache : p.k_cache) + ((static_cast<size_t>(layer) * p.nkv + g) * p.max_context + sh.n_old) * D + i;
            d[0] = f32_to_bf16_bits(lo);
            d[half] = f32_to_bf16_bits(hi);
        }
    } else if (op == ST_GU) {
        put1(p.act_ll + j, lo / (1.f + expf(-lo)) * hi, tag);
    } else if (op == ST_LM) {
        float *logits = p.req->logits_out;
        if (logits) logits[j] = lo;
        if (arg_better(lo, j, best_v, best_i)) { best_v = lo; best_i = j; }
    } else {
        const float resid = c.resid()[j - u0] += lo;
        put1((op == ST_O ? p.xo_ll : p.x_ll) + static_cast<size_t>(c.cta) * p.x_line + (j - u0), resid, tag);
    }
}

__device__ __forceinline__ void arg_fold(float &v, int &i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (arg_better(ov, oi, v, i)) { v = ov; i = oi; }
    }
}

template <int D, int G, bool Q8>
__global__ void __launch_bounds__(ST_THREADS, 1) step_kernel(const __grid_constant__ StepParams p) {
    Ctx c(p);
    {
        Shared &sh = c.sh();
        const uint4 *src = reinterpret_cast<const uint4 *>(p.layers);
        uint4 *dst = reinterpret_cast<uint4 *>(st_smem + ST_SHARED_BYTES + p.ring_bytes);
        for (int i = c.tid; i < (p.n_layers + 1) * 4; i += ST_THREADS) dst[i] = src[i];
        if (c.tid == 0) {
            for (int i = 0; i < ST_BARS; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], ST_NW); }
            sh.abort = 0;
            sh.sent = 0u;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            const int rt = p.req->token, rp = p.req->position;
            sh.token = rt >= 0 ? rt : p.state->next_token;
            sh.pos = rp >= 0 ? rp : p.state->next_position;
            sh.n_old = p.state->cur_len;
            sh.tag0 = static_cast<unsigned>(p.state->reserved[0]) * static_cast<unsigned>(p.n_layers + 2) + 1u;
            sh.odd = static_cast<unsigned>(p.barrier_extra) << 31;
            sh.total_x = c.ncta * line_units(p.H, c.ncta, 1);
            sh.total_a = c.ncta * line_units(p.qd, c.ncta, 2);
        }
        __syncthreads();
        const int lm_rows = c.head().rows;
        // a corrupt request or state: compute nothing
        if (sh.token < 0 || sh.token >= p.V || sh.n_old < 0 || sh.n_old >= p.max_context || sh.pos < 0 || lm_rows < 1 || lm_rows > p.V) {
            if (c.tid == 0 && atomicCAS(&p.state->status, 0, 103) == 0) { p.state->pad[0] = sh.token; p.state->pad[1] = sh.n_old; }
            return;
        }
        if (c.tid < 5) {
            const int n = op_units(p, c.tid, lm_rows);
            sh.u0[c.tid] = st_first(n, c.cta, c.ncta);
            sh.u1[c.tid] = st_first(n, c.cta + 1, c.ncta);
        }
        if (c.tid == 32) sh.share = kv_share(p, sh.n_old, c.cta, c.ncta);
        __syncthreads();                 // the last sync of all threads
    }
    if (c.warp >= ST_NW) {               // the feeding warpgroup: gives its registers to the others
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(ST_REGS_FEED));
        if (c.warp == ST_NW && c.lane == 0) feed_ring<Q8>(c);
        if (c.warp == ST_NW + 1 && c.lane == 0) feed_l2<Q8>(c);
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(ST_REGS));
    constexpr int half = D / 2;
    int prof_idx = 0;
    stamp(c, prof_idx);
    // The small per-layer vectors are read on the critical path right behind an exchange: ask L2 for all of them now (they stay, the
    // weight stream is evict-first).
    {
        const int lines_h = (p.H + 63) / 64, lines_q = ((p.nq + 2 * p.nkv) * D + 63) / 64, per_layer = 2 * lines_h + lines_q;
#pragma unroll 1
        for (int i = c.cta * ST_NT + c.tid; i < p.n_layers * per_layer + lines_h; i += c.ncta * ST_NT) {
            const int layer = i / per_layer, l = i - layer * per_layer;
            const StepLayer *L = c.layer(layer);
            const uint16_t *v = layer == p.n_layers ? c.head().final_norm + 64 * l
                                : l < lines_h ? L->input_norm + 64 * l : l < 2 * lines_h ? L->post_norm + 64 * (l - lines_h)
                                : L->bqkv ? L->bqkv + 64 * (l - 2 * lines_h) : nullptr;
            if (v) asm volatile("prefetch.global.L2 [%0];" ::"l"(v));
        }
    }
    {
        Shared &sh = c.sh();
        for (int i = c.tid; i < half; i += ST_NT) {        // rotary table of the step's position; fp64 angle, rounded once
            double sn, cs;
            sincos(static_cast<double>(sh.pos) * p.inv_freq[i], &sn, &cs);
            sh.rope[i] = static_cast<float>(cs);
            sh.rope[half + i] = static_cast<float>(sn);
        }
        if (c.cta == 0 && c.tid == 0) { p.state->token = sh.token; p.state->position = sh.pos; }
        make_table(c, c.unit_table(), p.H, 1, p.x_line);
        make_table(c, c.unit_table() + sh.total_x, p.qd, 2, p.ao_line);
        const uint16_t *erow = p.embed + static_cast<size_t>(sh.token) * p.H;
        const int x0 = sh.u0[ST_DN], x1 = sh.u1[ST_DN];
        for (int i = c.tid; i < x1 - x0; i += ST_NT) c.resid()[i] = bf16_bits_to_f32(erow[x0 + i]);
    }
    float best_v = -INFINITY;
    int best_i = 0x7fffffff;
    unsigned batch = 0;
    bool ok = cta_vote(true);            // tables

#pragma unroll 1
    for (int ph = 0; ph <= 4 * p.n_layers && ok; ++ph) {
        const int layer = ph >> 2;
        int op = layer == p.n_layers ? ST_LM : ph & 3;
        // one copy of the loop body, not one per operator, and no address carried in registers from one operator to the next
        asm volatile("" : "+r"(op), "+r"(c.tid), "+r"(c.cta), "+r"(c.ncta));
        c.warp = c.tid >> 5;
        c.lane = c.tid & 31;
        Shared &sh = c.sh();
        const unsigned tag = (sh.tag0 + static_cast<unsigned>(layer)) ^ sh.odd;      // what this layer's packets are expected to carry
        const StepLayer *L = c.layer(layer);
        // -- the input vector --
        if (op == ST_O) {
            stamp(c, prof_idx);
            if (sh.share.any) ok = attend<D, G, Q8>(c, layer, tag);
            if (!ok) break;
            stamp(c, prof_idx);                       // chunk done
            ok = merge_chunks(c, tag);
            if (!ok) break;
            stamp(c, prof_idx);                       // partial results merged
        }
        if (op == ST_QKV && layer == 0) {
            ok = stage_embedding(c, L->input_norm);
        } else if (op != ST_DN) {                     // (one call for the three exchanges: the loop's code has to stay small)
            const bool ao = op == ST_O, gu = op == ST_GU;
            ok = stage_lines(c, c.unit_table() + (ao ? sh.total_x : 0), ao ? sh.total_a : sh.total_x, (ao ? p.qd : p.H) / 8, ao ? p.ao_ll : gu ? p.xo_ll : p.x_ll,
                             ao ? nullptr : gu ? L->post_norm : op == ST_QKV ? L->input_norm : c.head().final_norm,
                             ao || gu ? tag : (sh.tag0 + static_cast<unsigned>(layer) - 1u) ^ sh.odd);
        }
        if (!ok) break;
        if (op == ST_DN) ok = stage_slice(c, p.act_ll, tag);       // (of this warp; the vote follows the products)
        stamp(c, prof_idx);
        // -- products, batch by batch, and their epilogues --
        const int u0 = sh.u0[op], u1 = sh.u1[op], per_batch = units_per_batch(op);
#pragma unroll 1
        for (int ub = u0; ub == u0 || ub < u1; ub += per_batch) {
            const int ue = min(u1, ub + per_batch), j = ub + c.tid;
            float add_lo = 0.f, add_hi = 0.f;          // biases, fetched ahead
            if (op == ST_QKV && L->bqkv && j < ue) {
                const int row = (j >> p.half_shift) * D + (j & (half - 1));
                add_lo = bf16_bits_to_f32(__ldg(L->bqkv + row));
                add_hi = bf16_bits_to_f32(__ldg(L->bqkv + row + half));
            }
            ok = ok && multiply_any(c, Slice{ub, ue, op, static_cast<int>(batch & 1u)});
            ok = cta_vote(ok);
            if (!ok) break;
            const float *a = sh.part[batch & 1u] + c.tid * ST_NW, *b = a + ST_BATCH * ST_NW;
            ++batch;
            if (j < ue) {
                float lo = 0.f, hi = 0.f;
#pragma unroll
                for (int w = 0; w < ST_NW; ++w) lo += a[w];
                if (op_paired(op)) {
#pragma unroll
                    for (int w = 0; w < ST_NW; ++w) hi += b[w];
                }
                finish_unit<D, Q8>(c, op, layer, j, u0, lo, hi, add_lo, add_hi, best_v, best_i);
            }
        }
        stamp(c, prof_idx);
        if (op != ST_QKV && op != ST_LM) stamp(c, prof_idx);
    }
    Shared &sh = c.sh();
    if (!ok) {
        *c.abort() = 1;
        if (c.tid == 0) atomicCAS(&p.state->status, 0, 6);
        return;
    }
    // ---- greedy token: thread -> CTA -> CTA 0 -> state --------------------------------------------------------------------
    arg_fold(best_v, best_i);
    if (c.lane == 0) { sh.best_v[c.warp] = best_v; sh.best_i[c.warp] = best_i; }
    cta_vote(true);
    const unsigned tag = sh.tag0 + static_cast<unsigned>(p.n_layers);
    if (c.tid == 0) {
        for (int w = 1; w < ST_NW; ++w)
            if (arg_better(sh.best_v[w], sh.best_i[w], best_v, best_i)) { best_v = sh.best_v[w]; best_i = sh.best_i[w]; }
        put2(p.lm_ll + static_cast<size_t>(c.cta) * 16, best_v, __int_as_float(best_i), tag);
    }
    if (c.cta != 0 || c.warp != 0) return;
    best_v = -INFINITY;
    best_i = 0x7fffffff;
    for (int i = c.lane; i < c.ncta && ok; i += 32) {
        Two t = get2(p.lm_ll + static_cast<size_t>(i) * 16);
        Spin sp;
        while (ok && !both(t, tag)) {
            ok = sp.again(c.abort(), p.spin_limit);
            t = get2(p.lm_ll + static_cast<size_t>(i) * 16);
        }
        const float v = packet_value(t.a);
        const int ix = __float_as_int(packet_value(t.b));
        if (arg_better(v, ix, best_v, best_i)) { best_v = v; best_i = ix; }
    }
    if (!__all_sync(0xffffffffu, ok)) {
        if (c.lane == 0) atomicCAS(&p.state->status, 0, 6);
        return;
    }
    arg_fold(best_v, best_i);
    if (c.lane == 0) {
        if (best_i < 0 || best_i >= c.head().rows) best_i = 0;       // (no logit compared as larger than -inf)
        if (c.head().remap) best_i = p.vocab_ids[best_i];
        if (p.req->next_token_out) *p.req->next_token_out = best_i;
        if (p.req->n_accepted_out) *p.req->n_accepted_out = 1;
        StepState *st = p.state;
        st->next_token = best_i;
        st->next_position = sh.pos + 1;
        st->cur_len = sh.n_old + 1;
        st->n_accepted = 1;
        st->reserved[0] += 1;
    }
}

template <int D, bool Q8>
StepKernel kernel_for(int G) {
    switch (G) {
        case 1: return step_kernel<D, 1, Q8>;
        case 2: return step_kernel<D, 2, Q8>;
        case 3: return step_kernel<D, 3, Q8>;
        case 4: return step_kernel<D, 4, Q8>;
        case 5: return step_kernel<D, 5, Q8>;
        case 6: return step_kernel<D, 6, Q8>;
        case 7: return step_kernel<D, 7, Q8>;
        default: return step_kernel<D, 8, Q8>;
    }
}

}  // namespace step
}  // namespace edgefm
