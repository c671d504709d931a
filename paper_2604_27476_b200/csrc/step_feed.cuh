// The weight stream of the decode-step kernel: the order of its chunks, the ring, the L2 look-ahead.
#pragma once
#include "step_prims.cuh"

namespace edgefm {
namespace step {

// Calls f(part) for every chunk of the whole step in order, until f returns false.  A chunk is one or two parts of `rows` segments of
// `seg` bytes, `stride` bytes apart in memory and packed in the ring (p1 null: one part).  Run by whole warps: the lanes share out the
// copies.
// With a tensor map: boxes at (0, row, block) and, for pairs, (0, row1, block) of `seg` bytes each.
struct Part { const unsigned char *p0, *p1; int rows; unsigned seg, stride; bool kv; const unsigned char *map; int row, row1, block; };
template <bool Q8, int MT, typename F>
__device__ __forceinline__ void for_each_chunk(const Ctx<MT> &c, F f) {
    const Shared<MT> &sh = c.sh();
    const StepParams &p = c.p();
    const int half = 1 << p.half_shift;
#pragma unroll 1
    for (int layer = 0; layer <= p.n_layers; ++layer) {
#pragma unroll 1
        for (int op = layer == p.n_layers ? ST_LM : ST_QKV; op <= (layer == p.n_layers ? ST_LM : ST_DN); ++op) {
            if (op == ST_O) {                                   // the cache rows come between the QKV and the O rows
                constexpr int E = Q8 ? 1 : 2;
#pragma unroll 1
                for (int idx = c.cta; idx < sh.m * p.nkv * sh.n_chunks; idx += c.ncta) {
                    const KvShare share = kv_share(p, sh.n_old, sh.n_chunks, idx);
                    const size_t at = ((static_cast<size_t>(layer) * p.nkv + share.g) * p.max_context + share.t0) * (p.D * E);
                    Part t{reinterpret_cast<const unsigned char *>(p.k_cache) + at, reinterpret_cast<const unsigned char *>(p.v_cache) + at, 1, 0u, 0u, true, nullptr, 0, 0, 0};
#pragma unroll 1
                    for (int pos = share.t0; pos < share.t1; pos += ST_KV_BLOCK) {
                        t.seg = static_cast<unsigned>(min(ST_KV_BLOCK, share.t1 - pos) * p.D * E);
                        if (!f(t)) return;
                        t.p0 += t.seg;
                        t.p1 += t.seg;
                    }
                }
            }
            const StepLayer *L = c.layer(layer);
            const unsigned char *w = reinterpret_cast<const unsigned char *>(op == ST_QKV ? L->wqkv : op == ST_O ? L->wo : op == ST_GU ? L->w_gate_up
                                                                             : op == ST_DN ? L->w_down : c.head().lm_head);
            const unsigned row_bytes = static_cast<unsigned>(p.cols[op].K) * 2u, seg = static_cast<unsigned>(p.cols[op].seg) * 2u;
            const int u0 = sh.u0[op], u1 = sh.u1[op];
            const bool paired = op_paired(op), whole = seg == row_bytes;
            const size_t partner = static_cast<size_t>(op == ST_QKV ? half : p.F) * row_bytes;
            w += static_cast<size_t>(op == ST_QKV ? (u0 >> p.half_shift) * p.D + (u0 & (half - 1)) : u0) * row_bytes;
#pragma unroll 1
            for (int u = u0; u < u1;) {
                const int n = tile_units(p, op, u, u1);
                Part t{w, paired ? w + partner : nullptr, whole ? 1 : n, whole ? static_cast<unsigned>(n) * row_bytes : seg, row_bytes, false, nullptr, 0, 0, 0};
                if (whole) {
                    if (!f(t)) return;
                } else if (p.cols[op].box_rows) {
                    t.map = p.maps + static_cast<size_t>(4 * layer + (op == ST_LM ? 0 : op)) * 128;
                    t.rows = 1;
                    t.seg = seg * static_cast<unsigned>(p.cols[op].box_rows);
                    t.row = op == ST_QKV ? (u >> p.half_shift) * p.D + (u & (half - 1)) : u;
                    t.row1 = t.row + (op == ST_QKV ? half : p.F);
#pragma unroll 1
                    for (int k = p.cols[op].segs; k > 0; --k) {
                        if (!f(t)) return;
                        t.block += p.cols[op].seg >> 6;
                    }
                } else {
#pragma unroll 1
                    for (unsigned at = 0; at < row_bytes; at += seg) {
                        t.seg = min(seg, row_bytes - at);
                        if (!f(t)) return;
                        t.p0 += seg;
                        if (paired) t.p1 += seg;
                    }
                }
                w += static_cast<size_t>(n) * row_bytes;
                u += n;
                if (op == ST_QKV && (u & (half - 1)) == 0) w += partner;                    // past the partner rows of the head just finished
            }
        }
    }
}

// One warp fills the ring ...
template <bool Q8, int MT>
__device__ __forceinline__ void feed_ring(Ctx<MT> &c) {
    Shared<MT> &sh = c.sh();
    const StepParams &p = c.p();
    unsigned long long once, keep;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(once));    // weights are read once per step
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(keep));
    const unsigned ring = static_cast<unsigned>(p.ring_bytes), limit = p.spin_limit, ring_at = smem_u32(c.ring());
    unsigned issued = 0, freed = 0;              // chunks copied / released so far
    unsigned at = 0, tail = 0;                   // next offset; start of the oldest chunk still in use
    unsigned sent = 0;                           // 16-byte units copied so far
    const unsigned char *fenced = nullptr;
    bool ok = true;
    for_each_chunk<Q8>(c, [&](const Part &t) {
        const unsigned part = static_cast<unsigned>(t.rows) * t.seg, bytes = t.p1 ? 2 * part : part, need = (bytes + 127u) & ~127u;
        // room: chunks lie one behind the other and are never cut; the oldest are waited for until this one fits
        for (;;) {
            if (issued == freed) { at = 0; tail = 0; break; }
            if (issued - freed < ST_BARS) {
                if (at >= tail) {
                    if (ring - at >= need) break;
                    if (tail > need) { at = 0; break; }
                } else if (tail - at > need) break;
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.empty[freed & (ST_BARS - 1)], (freed / ST_BARS) & 1u, c.abort(), limit))) { ok = false; return false; }
            ++freed;
            tail = freed == issued ? at : *reinterpret_cast<volatile unsigned *>(&sh.chunk_at[freed & (ST_BARS - 1)]);
        }
        const unsigned b = issued & (ST_BARS - 1), bar = smem_u32(&sh.full[b]);
        if (c.lane == 0) {
            *reinterpret_cast<volatile unsigned *>(&sh.chunk_at[b]) = at;
            mbar_expect_tx(&sh.full[b], bytes);
        }
        __syncwarp();
        const int r = c.lane & 15;
        if (t.map) {
            if (c.lane == 0 && (p.map_fence == 2 || (p.map_fence == 1 && t.map == p.maps + static_cast<size_t>(4 * p.n_layers) * 128)) && t.map != fenced) {
                // order the copy engine's view of a map the host may have rewritten behind what is in memory now
                fenced = t.map;
                asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(t.map) : "memory");
            }
            if (c.lane == 0)
                asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(ring_at + at),
                             "l"(t.map), "r"(0), "r"(t.row), "r"(t.block), "r"(bar), "l"(once)
                             : "memory");
            if (c.lane == 0 && t.p1)
                asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(ring_at + at + part),
                             "l"(t.map), "r"(0), "r"(t.row1), "r"(t.block), "r"(bar), "l"(once)
                             : "memory");
        } else if (r < t.rows && (c.lane < 16 || t.p1)) {
            const unsigned char *src = (c.lane < 16 ? t.p0 : t.p1) + static_cast<size_t>(r) * t.stride;
            const unsigned dst = ring_at + at + (c.lane < 16 ? 0u : part) + static_cast<unsigned>(r) * t.seg;
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst), "l"(src), "r"(t.seg),
                         "r"(bar), "l"(t.kv ? keep : once)
                         : "memory");
        }
        at += need;
        ++issued;
        sent += bytes >> 4;
        if (c.lane == 0) *reinterpret_cast<volatile unsigned *>(&sh.sent) = sent;
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
template <bool Q8, int MT>
__device__ __forceinline__ void feed_l2(Ctx<MT> &c) {
    Shared<MT> &sh = c.sh();
    const unsigned ahead = static_cast<unsigned>(c.p().prefetch_bytes) >> 4;
    if (ahead == 0) return;
    unsigned pos = 0;
    for_each_chunk<Q8>(c, [&](const Part &t) {
        pos += (static_cast<unsigned>(t.rows) * t.seg * (t.p1 ? 2 : 1)) >> 4;
        unsigned spins = 0;
        int lead;                                // (differences: the counters may wrap)
        while ((lead = static_cast<int>(pos - __shfl_sync(0xffffffffu, *reinterpret_cast<volatile unsigned *>(&sh.sent), 0))) > static_cast<int>(ahead)) {
            if (__any_sync(0xffffffffu, *c.abort()) || ++spins > (1u << 22)) return false;      // bounded; a hint not given costs only time
            __nanosleep(64);
        }
        if (lead <= 0) return true;              // the ring has it already
        const int r = c.lane & 15;
        if (t.map) {
            if (c.lane == 0 && c.p().map_fence != 2 && t.map != c.p().maps + static_cast<size_t>(4 * c.p().n_layers) * 128) {   // (only through maps that are never rewritten)
                asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(t.map), "r"(0), "r"(t.row), "r"(t.block) : "memory");
                if (t.p1) asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(t.map), "r"(0), "r"(t.row1), "r"(t.block) : "memory");
            }
        } else if (r < t.rows && (c.lane < 16 || t.p1))
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((c.lane < 16 ? t.p0 : t.p1) + static_cast<size_t>(r) * t.stride), "r"(t.seg) : "memory");
        return true;
    });
}

// A third warp brings the vectors: when all CTAs have arrived, one bulk copy (they lie in memory as they are wanted in shared memory).
// MLP activations come segment by segment, a few ahead of the products.  That a copy may overwrite the area follows from this CTA's
// own arrival: it comes after the last read of what was there.
template <int MT>
__device__ __forceinline__ void feed_vectors(Ctx<MT> &c) {
    Shared<MT> &sh = c.sh();
    const StepParams &p = c.p();
    constexpr int NA = Ctx<MT>::NA;
    unsigned k = 0, target = static_cast<unsigned>(p.state->epoch[p.epoch_slot]) * static_cast<unsigned>((st_packets(MT) ? 1 : 4) * p.n_layers * c.ncta) + static_cast<unsigned>(p.barrier_extra);
    bool ok = true;
    auto everybody = [&]() {                     // wait for the next exchange's arrivals
        target += static_cast<unsigned>(c.ncta);
        Spin sp;
        for (;;) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p.arrivals) : "memory");
            if (static_cast<int>(v - target) >= 0) break;
            if (!sp.again(c.abort(), p.spin_limit)) return false;
        }
        asm volatile("fence.proxy.async;" ::: "memory");
        return true;
    };
    auto copy = [&](const unsigned char *from, unsigned to, int bytes) {
        unsigned long long *bar = &sh.x_full[k & 3u];
        mbar_expect_tx(bar, static_cast<unsigned>(bytes));
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(c.area()) + to), "l"(from), "r"(bytes),
                     "r"(smem_u32(bar))
                     : "memory");
        ++k;
    };
    const int vec = NA * st_array_bytes(p.H) + 4 * MT * p.ss_stride, slot = NA * st_array_bytes(p.cols[ST_DN].seg), segs = p.cols[ST_DN].segs;
    const int tiles = (sh.u1[ST_DN] - sh.u0[ST_DN] + ST_TILE - 1) / ST_TILE;
#pragma unroll 1
    for (int layer = 0; layer <= p.n_layers && ok; ++layer) {
        if constexpr (!st_packets(MT)) {
            if (layer > 0) {
                ok = everybody();
                if (ok) copy(p.x_vec, 0u, vec);
            }
            if (!ok || layer == p.n_layers) break;
            ok = everybody();
            if (!ok) break;
            copy(p.ao_vec, 0u, NA * st_array_bytes(p.qd));
            ok = everybody();
            if (!ok) break;
            copy(p.xo_vec, 0u, vec);
        }
        if (layer == p.n_layers) break;
        ok = everybody();
        if (!ok) break;
        const unsigned first = k;
#pragma unroll 1
        for (int i = 0; i < tiles * segs && ok; ++i) {
            const unsigned back = k - static_cast<unsigned>(p.act_slots);
            if (k - first >= static_cast<unsigned>(p.act_slots)) ok = mbar_wait(&sh.x_empty[back & 3u], (back >> 2) & 1u, c.abort(), p.spin_limit);
            if (ok) copy(p.act_vec + static_cast<size_t>(i % segs) * slot, static_cast<unsigned>(i % p.act_slots) * slot, slot);
        }
    }
    if (!ok) {               // giving up: the copies in flight must land before the CTA's shared memory is released
        int dummy = 0;
        for (unsigned j = k > 4 ? k - 4 : 0; j < k; ++j) mbar_wait(&sh.x_full[j & 3u], (j >> 2) & 1u, &dummy, p.spin_limit);
    }
}

}  // namespace step
}  // namespace edgefm
