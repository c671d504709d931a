// The whole decode step as ONE persistent cooperative kernel (one CTA per SM): every warp owns a slice of the COLUMNS.
//
// At batch 1 a step is a chain of matrix-vector products bound by the one pass over the weights, but cut by six exchanges per
// layer in which every SM needs what the others computed.  Two things decide its time: that the weight stream never stops,
// and what an exchange costs.
//
//   * Weights (step_feed.cuh).  A CTA owns a contiguous range of the rows of every operator, i.e. a contiguous range of memory.
//     One thread feeds a ring in shared memory with bulk copies (cp.async.bulk, up to 68 KB each) in the order of the whole step --
//     QKV rows, this CTA's K/V cache rows, O rows, gate/up rows, down rows, next layer, ..., output layer -- independent of the
//     computation; another asks L2 for what comes after the ring.  (A bulk copy costs its issuer the same few hundred cycles
//     whatever its size: measured from L2, 6 / 24 / 48 KB copies from one such loop reached 2.2 / 9 / 18 TB/s over the chip.)
//   * Products (step_products.cuh).  All 8 consumer warps work on every tile of 16 rows (or 8 row pairs); warp w multiplies its share of
//     the columns on the tensor cores, mma.m16n8k16 as a dot-product unit: the activations enter as bf16 pieces (three for one or
//     two tokens, two for more), one B column per piece and token, so that a block of tokens costs the weights' traffic and the
//     instructions of one.  The 8 partial sums of a row meet in shared memory and one thread per output unit and token runs the
//     fused epilogue (bias + RoPE + cache row, residual add, SwiGLU, logits + argmax).
//   * Exchanges.  A value travels as an 8-byte packet with a tag that names step and layer, so a reader polls the data itself: one
//     trip to L2 instead of store, fence, counter, poll, load (a release waits for everything its SM has under way: 0.6 us idle,
//     2 us while the weights stream).  Vectors that are multiplied next travel as their bf16 pieces, split (and weighted for the norm)
//     once by the owner instead of by every reader.  Every CTA writes its values into 128-byte lines of its own (packets of several
//     writers in one line cost 0.3 - 1 us: the pollers' copies of the line are invalidated by every write); only the MLP activations
//     lie in natural order, with two writers in most lines where CTAs meet.
//     Polling grows with the tokens.  For four and more the owners write such vectors plainly, as the products want them, every CTA
//     counts up one counter, and a feeding thread that has seen all of them fetches the vector with one bulk copy (when
//     the two were compared a block of four took 1530 us with packets and 1286 us so, a single token 976 and 1016 us).  MLP activations too long for the shared memory go
//     this way too, by segments.  A buffer is rewritten one layer later; a CTA that writes it then has seen, in
//     between, an exchange to which every CTA contributes only after reading the old contents.
//   * Attention (step_attention.cuh).  CTA (token, kv head, chunk) holds the chunk's K/V rows in its ring before the queries exist,
//     serves the whole GQA group from one read, and publishes unnormalised partial results; the owner of an output pair merges
//     them (lanes over chunks) and publishes the finished vector.  The rows this call appends travel as packets too.
//   * Several tokens (Sec. 3.11 of the paper: the base model verifies a proposed block): tokens[0] and the proposed continuation pass
//     through the step together, at consecutive positions and cache slots; CTA 0 accepts the longest prefix that greedy decoding
//     would have produced.
//
// Every wait is bounded: on expiry the CTA records STATUS_TIMEOUT and all its warps leave at the next CTA-wide vote; the feeding threads
// leave when their copies have landed (bounded, too).
#include "step_attention.cuh"
#include "step_feed.cuh"
#include "step_products.cuh"

namespace edgefm {
namespace ST_NS {

// The epilogue of output unit j of token `tok` (its row sum, or the sums of its two rows) of the QKV, gate/up and output layer operators.
template <int D, bool Q8, int MT>
__device__ __forceinline__ void finish_unit(const Ctx<MT> &c, int op, int layer, int tok, int j, int u0, float lo, float hi, float add_lo, float add_hi, float &best_v,
                                            int &best_i) {
    const Shared<MT> &sh = c.sh();
    const StepParams &p = c.p();
    constexpr int half = D / 2;
    const unsigned tag = sh.tag0 + static_cast<unsigned>(layer);
    if (op == ST_QKV) {
        const int head = j >> p.half_shift, i = j & (half - 1);
        lo += add_lo;
        hi += add_hi;
        if (head < p.nq + p.nkv) {
            const float cs = sh.rope[tok][i], sn = sh.rope[tok][half + i];
            const float a = lo * cs - hi * sn, b = hi * cs + lo * sn;
            lo = a;
            hi = b;
        }
        put2(p.q_ll + (static_cast<size_t>(tok) * c.ncta + c.cta) * p.q_line + 2 * (j - u0), lo, hi, tag);
        if (!Q8 && head >= p.nq && tok < sh.m) {
            const bool is_v = head >= p.nq + p.nkv;
            const int g = head - p.nq - (is_v ? p.nkv : 0);
            uint16_t *d = (is_v ? p.v_cache : p.k_cache) + ((static_cast<size_t>(layer) * p.nkv + g) * p.max_context + sh.n_old + tok) * D + i;
            d[0] = f32_to_bf16_bits(lo);
            d[half] = f32_to_bf16_bits(hi);
        }
    } else if (op == ST_GU) {
        const float v = lo / (1.f + expf(-lo)) * hi;
        if (st_packets(MT) && p.act_packets) {
            put_raw(p.act_ll + static_cast<size_t>(tok) * p.act_len + j, pieces_packet(v, tag));
            return;
        }
        const int seg = p.cols[ST_DN].seg, s = j / seg, stride = st_array_bytes(seg);
        store_pieces<MT>(p.act_vec + static_cast<size_t>(s) * Ctx<MT>::NA * stride, tok, j - s * seg, stride, v);
    } else if (tok < sh.m) {
        float *logits = p.req.logits_out;
        if (logits) logits[static_cast<size_t>(tok) * c.head().rows + j] = lo;
        if (arg_better(lo, j, best_v, best_i)) { best_v = lo; best_i = j; }
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

template <int D, int G, bool Q8, int MT>
__global__ void __launch_bounds__(ST_THREADS, 1) step_kernel(const __grid_constant__ StepParams p) {
    Ctx<MT> c(p);
    {
        Shared<MT> &sh = c.sh();
        const uint4 *src = reinterpret_cast<const uint4 *>(p.layers);
        uint4 *dst = reinterpret_cast<uint4 *>(st_smem + st_shared_bytes<MT>() + p.ring_bytes);
        for (int i = c.tid; i < (p.n_layers + 1) * 4; i += ST_THREADS) dst[i] = src[i];
        if (c.tid == 0) {
            for (int i = 0; i < ST_BARS; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], ST_NW); }
            for (int i = 0; i < 4; ++i) { mbar_init(&sh.x_full[i], 1); mbar_init(&sh.x_empty[i], ST_NW); }
            sh.abort = 0;
            sh.sent = 0u;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            const int rt = p.req.token, rp = p.req.position, st_token = p.state->next_token, st_pos = p.state->next_position, st_len = p.state->cur_len, st_status = p.state->status;
            const unsigned epoch = static_cast<unsigned>(p.state->epoch[p.epoch_slot]);
            sh.m = MT > 1 ? min(max(p.req.m, 1), MT) : 1;
            sh.tokens[0] = rt >= 0 ? rt : st_token;
            for (int t = 1; t < MT; ++t) sh.tokens[t] = t < sh.m ? p.req.draft[t - 1] : 0;
            sh.pos = rp >= 0 ? rp : st_pos;
            sh.n_old = st_status == STATUS_TIMEOUT ? -1 : st_len;
            sh.n_chunks = kv_chunks(p, sh.n_old, sh.m, c.ncta);
            sh.tag0 = epoch * static_cast<unsigned>(p.n_layers + 2) + 1u;
            sh.odd = static_cast<unsigned>(p.barrier_extra) << 31 | static_cast<unsigned>(p.barrier_extra) << 15;
            sh.total_x = c.ncta * line_units(p.H, c.ncta, 1);
            sh.total_a = c.ncta * line_units(p.qd, c.ncta, 2);
        }
        __syncthreads();
        const int lm_rows = c.head().rows;
        bool sane = true;
        for (int t = 0; t < MT; ++t) sane = sane && sh.tokens[t] >= 0 && sh.tokens[t] < p.V;
        // a corrupt request or state, or an earlier step that ran into the bound of a wait: compute nothing
        if (!sane || sh.n_old < 0 || sh.n_old + sh.m > p.max_context || sh.pos < 0 || lm_rows < 1 || lm_rows > p.V) {
            if (c.tid == 0 && atomicCAS(&p.state->status, 0, 103) == 0) { p.state->pad[0] = sh.tokens[0]; p.state->pad[1] = sh.n_old; }
            return;
        }
        if (c.tid < 5) {
            const int n = op_units(p, c.tid, lm_rows);
            sh.u0[c.tid] = st_first(n, c.cta, c.ncta);
            sh.u1[c.tid] = st_first(n, c.cta + 1, c.ncta);
        }
        __syncthreads();                 // the last sync of all threads
    }
    if (c.warp >= ST_NW) {               // the feeding warpgroup: gives its registers to the others
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(ST_REGS_FEED));
        if constexpr (!TIGHT) make_list(c);
        if (c.warp == ST_NW && c.lane == 0) feed_ring<Q8, MT>(c);
        if (c.warp == ST_NW + 1 && c.lane == 0) feed_l2<Q8, MT>(c);
        if (c.warp == ST_NW + 2 && c.lane == 0 && !(st_packets(MT) && p.act_packets)) feed_vectors<MT>(c);
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(ST_REGS));
    constexpr int half = D / 2, RB = Ctx<MT>::RB, RB_LOG2 = RB == 128 ? 7 : RB == 64 ? 6 : 5;
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
    const int x0 = c.sh().u0[ST_DN], my_rows = c.sh().u1[ST_DN] - x0;      // rows of the residual stream this CTA owns
    {
        Shared<MT> &sh = c.sh();
        // warps 0 .. rw - 1 make the rotary tables of the tokens' positions (fp64 angle, rounded once), the others the unit tables
        const int rw = st_packets(MT) ? MT * half / 32 : ST_NW;
        for (int i = c.tid; i < sh.m * half && c.warp < rw; i += rw * 32) {
            const int t = i / half, f = i - t * half;
            double sn, cs;
            sincos(static_cast<double>(sh.pos + t) * p.inv_freq[f], &sn, &cs);
            sh.rope[t][f] = static_cast<float>(cs);
            sh.rope[t][half + f] = static_cast<float>(sn);
        }
        if (c.cta == 0 && c.tid == 0) { p.state->token = sh.tokens[0]; p.state->position = sh.pos; }
        if constexpr (st_packets(MT) && !TIGHT) {
            const int threads = (ST_NW - rw) * 32, first = c.tid - rw * 32;
            if (first >= 0) {
                make_table(c, c.unit_table(), p.H, 1, p.x_line, first, threads);
                make_table(c, c.unit_table() + sh.total_x, p.qd, 2, p.ao_line, first, threads);
            }
        }
    }
    float best_v = -INFINITY;
    int best_i = 0x7fffffff;
    unsigned batch = 0;
    bool ok = true;

#pragma unroll 1
    for (int ph = 0; ph <= 4 * p.n_layers && ok; ++ph) {
        const int layer = ph >> 2;
        int op = layer == p.n_layers ? ST_LM : ph & 3;
        // one copy of the loop body, not one per operator, and no address carried in registers from one operator to the next
        asm volatile("" : "+r"(op), "+r"(c.tid), "+r"(c.cta), "+r"(c.ncta));
        c.warp = c.tid >> 5;
        c.lane = c.tid & 31;
        Shared<MT> &sh = c.sh();
        const unsigned real_tag = sh.tag0 + static_cast<unsigned>(layer), tag = real_tag ^ sh.odd;      // what this layer's packets carry / are expected to carry
        const StepLayer *L = c.layer(layer);
        // -- the input vector --
        if (op == ST_O) {
            stamp(c, prof_idx);
#pragma unroll 1
            for (int idx = c.cta; idx < sh.m * p.nkv * sh.n_chunks && ok; idx += c.ncta) {
                ok = attend<D, G, Q8, MT>(c, layer, kv_share(p, sh.n_old, sh.n_chunks, idx), tag);
                if (ok && idx + c.ncta < sh.m * p.nkv * sh.n_chunks) ok = cta_vote(true);
            }
            if (!ok) break;
            stamp(c, prof_idx);                       // chunk done
            ok = merge_chunks(c, tag);
            if constexpr (!st_packets(MT)) ok = arrive(c, ok);
            if (!ok) break;
            stamp(c, prof_idx);                       // partial results merged
        }
        if (op == ST_QKV && layer == 0) {
            ok = stage_embedding(c, L->input_norm, x0, my_rows);     // (its vote also publishes the tables)
        } else if (op == ST_DN) {
            c.act_slot = 0;
            if (st_packets(MT) && p.act_packets) ok = stage_activations(c, tag);
        } else if constexpr (st_packets(MT)) {        // (one call for the three exchanges: the loop's code has to stay small)
            const bool ao = op == ST_O, gu = op == ST_GU;
            ok = stage_lines(c, (TIGHT ? p.unit_tab : c.unit_table()) + (ao ? sh.total_x : 0), ao ? sh.total_a : sh.total_x, ao ? p.qd : p.H, ao ? p.ao_ll : gu ? p.xo_ll : p.x_ll,
                             ao ? p.ao_line : p.x_line, !ao, ao || gu ? tag : (real_tag - 1u) ^ sh.odd);
        } else {
            ok = stage_vector(c, op != ST_O);         // (of this warp; the vote follows the products)
        }
        stamp(c, prof_idx);
        // -- products, batch by batch, and their epilogues --
        const int u0 = sh.u0[op], u1 = sh.u1[op];
        const bool paired = op_paired(op), resid = op == ST_O || op == ST_DN;
        const int batch_log2 = paired ? RB_LOG2 - 1 : RB_LOG2, per_batch = 1 << batch_log2;
        float sq = 0.f;                               // residual operators: this lane's share of the next norm's sum of squares
#pragma unroll 1
        for (int ub = u0, ue = u0, more = 1; more; ub = ue, more = ub < u1) {       // (once if the CTA owns nothing)
            ue = u1;                                   // a batch is whole tiles
            if (u1 - ub > per_batch) {
                ue = ub;
#pragma unroll 1
                for (int n; (n = tile_units(p, op, ue, u1)) <= per_batch - (ue - ub) && ue < u1;) ue += n;
            }
            // thread -> (token, unit): residual operators take a warp per token, lanes over rows
            const int tok = resid ? c.warp : c.tid >> batch_log2, j = ub + (resid ? c.lane : c.tid & (per_batch - 1));
            const bool mine = tok < MT && j < ue;
            float add_lo = 0.f, add_hi = 0.f;          // biases / the next norm's weight, fetched ahead
            if (mine) {
                if (op == ST_QKV && L->bqkv) {
                    const int row = (j >> p.half_shift) * D + (j & (half - 1));
                    add_lo = bf16_bits_to_f32(__ldg(L->bqkv + row));
                    add_hi = bf16_bits_to_f32(__ldg(L->bqkv + row + half));
                }
            }
            const uint16_t *next_norm = op == ST_O ? L->post_norm : layer + 1 == p.n_layers ? c.head().final_norm : c.layer(min(layer + 1, p.n_layers - 1))->input_norm;
            if (resid && mine) add_lo = bf16_bits_to_f32(__ldg(next_norm + j));
            ok = ok && multiply_any<MT>(c, Slice{ub, ue, op, static_cast<int>(batch & 1u)});
            ok = cta_vote(ok);
            if (!ok) break;
            const float *part = sh.part[batch & 1u];
            ++batch;
            if (resid) {
                if (tok < MT) {
                    unsigned char *vec = op == ST_O ? p.xo_vec : p.x_vec;
                    unsigned long long *line = (op == ST_O ? p.xo_ll : p.x_ll) + (static_cast<size_t>(tok) * c.ncta + c.cta) * p.x_line;
                    const int stride = st_array_bytes(p.H);
#pragma unroll 1
                    for (int r = j; r < ue; r += 32) {
                        if (r != j) add_lo = bf16_bits_to_f32(__ldg(next_norm + r));
                        float &x = c.resid()[tok * my_rows + r - u0];
                        x += sum8(part + (tok * RB + r - ub) * ST_NW);
                        sq = fmaf(x, x, sq);
                        if constexpr (st_packets(MT)) put_raw(line + r - u0, pieces_packet(x * add_lo, real_tag));
                        else store_pieces<MT>(vec, tok, r, stride, x * add_lo);
                    }
                    if (ue == u1) {
                        const float all = warp_sum(sq);
                        if (c.lane == 0 && st_packets(MT)) put1(line + p.x_line - 1, all, real_tag);
                        if (c.lane == 0 && !st_packets(MT)) *reinterpret_cast<float *>(vec + Ctx<MT>::NA * stride + 4 * (tok * p.ss_stride + c.cta)) = all;
                    }
                }
            } else if (mine) {
                const float r = rsqrtf(sh.ss[tok] / static_cast<float>(p.H) + p.eps);       // the deferred RMSNorm factor
                const float *a = part + (tok * RB + j - ub) * ST_NW;
                const float lo = sum8(a) * r, hi = paired ? sum8(a + RB / 2 * ST_NW) * r : 0.f;
                finish_unit<D, Q8, MT>(c, op, layer, tok, j, u0, lo, hi, add_lo, add_hi, best_v, best_i);
            }
        }
        stamp(c, prof_idx);
        if (ok && op != ST_QKV && op != ST_LM) {
            if (!st_packets(MT) || (op == ST_GU && !p.act_packets)) ok = arrive(c, true);
            stamp(c, prof_idx);
        }
    }
    Shared<MT> &sh = c.sh();
    if (!ok) {
        *c.abort() = 1;
        if (c.tid == 0) atomicExch(&p.state->status, STATUS_TIMEOUT);
        return;
    }
    // ---- greedy tokens: thread -> warp -> CTA -> CTA 0 -> state ------------------------------------------------------------
    // (threads tok * RB .. tok * RB + RB - 1 hold candidates of token tok: whole warps)
    arg_fold(best_v, best_i);
    if (c.lane == 0) { sh.best_v[c.warp] = best_v; sh.best_i[c.warp] = best_i; }
    cta_vote(true);
    const unsigned tag = sh.tag0 + static_cast<unsigned>(p.n_layers);
    constexpr int WT = RB / 32;          // warps per token
    if (c.tid < sh.m) {
        best_v = sh.best_v[c.tid * WT];
        best_i = sh.best_i[c.tid * WT];
        for (int w = 1; w < WT; ++w)
            if (arg_better(sh.best_v[c.tid * WT + w], sh.best_i[c.tid * WT + w], best_v, best_i)) { best_v = sh.best_v[c.tid * WT + w]; best_i = sh.best_i[c.tid * WT + w]; }
        put2(p.lm_ll + static_cast<size_t>(c.cta) * 16 + 2 * c.tid, best_v, __int_as_float(best_i), tag);
    }
    if (c.cta != 0) return;
    cta_vote(true);                      // (best_v / best_i have been read)
    best_v = -INFINITY;
    best_i = 0x7fffffff;
    if (c.warp < sh.m) {                 // warp t: token t
        for (int base = 0; base < c.ncta && ok; base += 32) {
            const int i = min(base + c.lane, c.ncta - 1);
            const unsigned long long *at = p.lm_ll + static_cast<size_t>(i) * 16 + 2 * c.warp;
            Two t;
            Spin sp;
            int more;
            do {
                t = get2(at);
                more = warp_again(sp, !both(t, tag), c.abort(), p.spin_limit);
            } while (more > 0);
            if (more == 0) { ok = false; break; }
            const float v = packet_value(t.a);
            const int ix = __float_as_int(packet_value(t.b));
            if (arg_better(v, ix, best_v, best_i)) { best_v = v; best_i = ix; }
        }
        arg_fold(best_v, best_i);
        if (c.lane == 0) {
            if (best_i < 0 || best_i >= c.head().rows) best_i = 0;       // (no logit compared as larger than -inf)
            if (c.head().remap) best_i = p.vocab_ids[best_i];
            sh.best_i[c.warp] = best_i;
        }
    }
    if (!cta_vote(ok)) {
        if (c.tid == 0) atomicExch(&p.state->status, STATUS_TIMEOUT);
        return;
    }
    if (c.tid == 0) {
        // Verification (Sec. 3.11): proposal t is accepted if it is the greedy choice after token t - 1; it stops at the first
        // rejection.  The cache advances by the accepted tokens; the rows of the rejected ones stay behind the cache length and are
        // overwritten by the next call.
        int n_acc = 1;
        const bool given = MT > 1 && (p.req.flags & 1);   // prompt tokens: nothing to verify
        while (n_acc < sh.m && (given || sh.tokens[n_acc] == sh.best_i[n_acc - 1])) ++n_acc;
        const int next = sh.best_i[n_acc - 1];
        if (p.req.next_token_out) *p.req.next_token_out = next;
        if (p.req.n_accepted_out) *p.req.n_accepted_out = n_acc;
        StepState *st = p.state;
        st->next_token = next;
        st->next_position = sh.pos + n_acc;
        st->cur_len = sh.n_old + n_acc;
        st->n_accepted = n_acc;
        st->epoch[p.epoch_slot] += 1;
    }
}

template <int D, bool Q8, int MT>
StepKernel kernel_for(int G) {
    switch (G) {
        case 1: return step_kernel<D, 1, Q8, MT>;
        case 2: return step_kernel<D, 2, Q8, MT>;
        case 3: return step_kernel<D, 3, Q8, MT>;
        case 4: return step_kernel<D, 4, Q8, MT>;
        case 5: return step_kernel<D, 5, Q8, MT>;
        case 6: return step_kernel<D, 6, Q8, MT>;
        case 7: return step_kernel<D, 7, Q8, MT>;
        default: return step_kernel<D, 8, Q8, MT>;
    }
}

}  // namespace ST_NS
}  // namespace edgefm
