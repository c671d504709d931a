// The weight stream of the decode-step kernel: the list of its chunks, the ring, the L2 look-ahead, the vectors.
#pragma once
#include "step_attention.cuh"

namespace edgefm {
namespace ST_NS {

// The order of the chunks is the same in every layer, so every CTA lists them once per launch (the feeding thread's time per chunk
// bounds the stream: with the addresses derived chunk by chunk it took about 1000 cycles from a freed slot to the next copy, and
// a ring of three 48 KB chunks delivered 9 instead of 17 TB/s from L2).  An entry:
//   x, y: first and second part, offset from the operator's matrix / 16 bytes (boxes: their first rows); y = ~0: one part
//   z: bytes of a part
//   w: 64-column block of a box | rows << 16, the row segments copied one by one (0: one copy; boxes: ST_BOX)
constexpr unsigned ST_BOX = 255u;
__host__ __device__ __forceinline__ uint4 chunk_entry(const StepParams &p, int op, int u, int n, int seg_i) {
    const StepCols &cols = p.cols[op];
    const int half = 1 << p.half_shift;
    const unsigned row = static_cast<unsigned>(op == ST_QKV ? (u >> p.half_shift) * p.D + (u & (half - 1)) : u), partner = row + static_cast<unsigned>(op == ST_QKV ? half : p.F);
    const bool paired = op_paired(op);
    const unsigned row16 = static_cast<unsigned>(cols.K) >> 3, at16 = static_cast<unsigned>(seg_i * cols.seg) >> 3;     // 16-byte units
    if (cols.segs == 1) return make_uint4(row * row16, paired ? partner * row16 : ~0u, static_cast<unsigned>(n) * row16 * 16u, 0u);
    if (cols.box_rows) return make_uint4(row, paired ? partner : ~0u, static_cast<unsigned>(cols.box_rows * cols.seg) * 2u, at16 >> 3 | ST_BOX << 16);
    return make_uint4(row * row16 + at16, paired ? partner * row16 + at16 : ~0u, min(static_cast<unsigned>(cols.seg) >> 3, row16 - at16) * 16u, static_cast<unsigned>(n) << 16);
}
// By the feeding warpgroup, for itself.
template <int MT> __device__ __forceinline__ void make_list(const Ctx<MT> &c) {
    constexpr int THREADS = ST_THREADS - ST_NT;
    const int tid = c.tid - ST_NT;
    Shared<MT> &sh = c.sh();
    const StepParams &p = c.p();
    // QKV tiles are cut at the ends of head halves, the others are regular
    int at = 0;
    for (int u = sh.u0[ST_QKV]; u < sh.u1[ST_QKV];) {
        const int n = tile_units(p, ST_QKV, u, sh.u1[ST_QKV]);
        for (int s = 0; s < p.cols[ST_QKV].segs; ++s, ++at)
            if (tid == at % THREADS) c.list()[at] = chunk_entry(p, ST_QKV, u, n, s);
        u += n;
    }
    for (int op = ST_O; op <= ST_LM; ++op) {
        const int tile = p.cols[op].tile, segs = p.cols[op].segs, u0 = sh.u0[op], u1 = sh.u1[op], count = (u1 - u0 + tile - 1) / tile * segs;
        if (tid == 0) sh.list[op] = at;
        for (int i = tid; i < count; i += THREADS) {
            const int k = i / segs, u = u0 + k * tile;
            c.list()[at + i] = chunk_entry(p, op, u, min(tile, u1 - u), i - k * segs);
        }
        at += count;
    }
    if (tid == 0) { sh.list[ST_QKV] = 0; sh.list[5] = at; }
    asm volatile("barrier.cta.sync 2, %0;" ::"n"(THREADS) : "memory");
}
// Calls f(base, entry, map) for the weights and f_kv(k, v, rows, bytes of each) for the cache rows of the whole step in order, until one returns false.
template <bool Q8, int MT, typename F, typename FKV>
__device__ __forceinline__ void for_each_chunk(const Ctx<MT> &c, F f, FKV f_kv) {
    const Shared<MT> &sh = c.sh();
    const StepParams &p = c.p();
    const uint4 *const list = c.list();
    constexpr int E = Q8 ? 1 : 2;
    const int block = kv_positions(p, p.D), row_bytes = p.D * E;
    const int shares = sh.m * p.nkv * sh.n_chunks;
    const unsigned char *map = p.maps;
#pragma unroll 1
    for (int layer = 0; layer <= p.n_layers; ++layer) {
        const bool lm = layer == p.n_layers;
        const StepLayer *L = c.layer(layer);
#pragma unroll 1
        for (int op = lm ? ST_LM : ST_QKV; op <= (lm ? ST_LM : ST_DN); ++op) {
            if (op == ST_O) {                                   // the cache rows come between the QKV and the O rows
#pragma unroll 1
                for (int idx = c.cta; idx < shares; idx += c.ncta) {
                    const KvShare share = kv_share(p, sh.n_old, sh.n_chunks, idx);
                    const size_t at = ((static_cast<size_t>(layer) * p.nkv + share.g) * p.max_context + share.t0) * (p.D * E);
                    const unsigned char *k = reinterpret_cast<const unsigned char *>(p.k_cache) + at, *v = reinterpret_cast<const unsigned char *>(p.v_cache) + at;
#pragma unroll 1
                    for (int pos = share.t0; pos < share.t1; pos += block) {
                        const int n = min(block, share.t1 - pos);
                        const unsigned bytes = static_cast<unsigned>(n * row_bytes);
                        if (!f_kv(k, v, n, bytes)) return;
                        k += bytes;
                        v += bytes;
                    }
                }
            }
            // (the first four pointers of a layer are its matrices in this order; the output layer's entry begins with its matrix)
            const unsigned char *base = lm ? reinterpret_cast<const unsigned char *>(c.head().lm_head)
                                           : reinterpret_cast<const unsigned char *>(reinterpret_cast<const uint16_t *const *>(L)[op]);
            if constexpr (TIGHT) {                              // (no list)
                int n;
#pragma unroll 1
                for (int u = sh.u0[op]; u < sh.u1[op]; u += n) {
                    n = tile_units(p, op, u, sh.u1[op]);
#pragma unroll 1
                    for (int seg = 0; seg < p.cols[op].segs; ++seg)
                        if (!f(base, chunk_entry(p, op, u, n, seg), map)) return;
                }
            } else {
                const int end = sh.list[op + 1];
#pragma unroll 1
                for (int i = sh.list[op]; i < end; ++i)
                    if (!f(base, list[i], map)) return;
            }
            map += 128;
        }
    }
}

// The last of a feeding thread's `issued` copies (`n` barriers, a power of two, used in turn) must land before the CTA's shared memory is
// released.  The products wait for them anyway, unless one has given up: then they may still be on their way when all other
// threads have left, whether the feeding thread had more to copy or not.  The bound is its own: the waits' may be shorter than a copy.
__device__ __forceinline__ void drain(unsigned long long *bars, unsigned n, unsigned issued) {
    int never = 0;
    for (unsigned k = issued > n ? issued - n : 0u; k < issued; ++k) mbar_wait(&bars[k & (n - 1u)], (k / n) & 1u, &never, ST_DRAIN_NS);
}

// One thread fills the ring ...
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
    const unsigned char *fenced = nullptr, *const lm_map = p.maps + static_cast<size_t>(4 * p.n_layers) * 128;
    bool ok = true;
    // room for a chunk: chunks lie one behind the other and are never cut; the oldest are waited for until this one fits.  Returns the
    // shared-memory address, and the barrier to complete on; 0: gave up.
    auto room = [&](unsigned bytes, unsigned space, unsigned &bar) {
        const unsigned need = (space + 127u) & ~127u;
        for (;;) {
            if (issued == freed) { at = 0; tail = 0; break; }
            if (issued - freed < ST_BARS) {
                if (at >= tail) {
                    if (ring - at >= need) break;
                    if (tail > need) { at = 0; break; }
                } else if (tail - at > need) break;
            }
            if (!mbar_wait(&sh.empty[freed & (ST_BARS - 1)], (freed / ST_BARS) & 1u, c.abort(), limit)) { ok = false; return 0u; }
            ++freed;
            tail = freed == issued ? at : *reinterpret_cast<volatile unsigned *>(&sh.chunk_at[freed & (ST_BARS - 1)]);
        }
        const unsigned b = issued & (ST_BARS - 1), to = ring_at + at;
        bar = smem_u32(&sh.full[b]);
        *reinterpret_cast<volatile unsigned *>(&sh.chunk_at[b]) = at;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        at += need;
        ++issued;
        sent += bytes >> 4;
        *reinterpret_cast<volatile unsigned *>(&sh.sent) = sent;
        return to;
    };
    auto bulk = [&](unsigned to, const unsigned char *from, unsigned bytes, unsigned bar, unsigned long long policy) {
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(to), "l"(from), "r"(bytes), "r"(bar), "l"(policy)
                     : "memory");
    };
    for_each_chunk<Q8>(
        c,
        [&](const unsigned char *base, const uint4 &e, const unsigned char *map) {
            const bool two = e.y != ~0u;
            const unsigned rows = e.w >> 16, part = e.z * (rows == 0u || rows == ST_BOX ? 1u : rows);
            unsigned bar;
            const unsigned all = two ? 2u * part : part, to = room(all, all, bar);
            if (!ok) return false;
            if (rows == 0u) {
                bulk(to, base + static_cast<size_t>(e.x) * 16u, part, bar, once);
                if (two) bulk(to + part, base + static_cast<size_t>(e.y) * 16u, part, bar, once);
            } else if (rows == ST_BOX) {
                if (map != fenced && (p.map_fence == 2 || (p.map_fence == 1 && map == lm_map))) {
                    // order the copy engine's view of a map the host may have rewritten behind what is in memory now
                    fenced = map;
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
                }
                asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(to), "l"(map),
                             "r"(0), "r"(e.x), "r"(e.w & 0xffffu), "r"(bar), "l"(once)
                             : "memory");
                if (two)
                    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(to + part),
                                 "l"(map), "r"(0), "r"(e.y), "r"(e.w & 0xffffu), "r"(bar), "l"(once)
                                 : "memory");
            } else {
                const size_t stride = static_cast<size_t>(p.cols[map == lm_map ? ST_LM : ((map - p.maps) >> 7) & 3].K) * 2;
#pragma unroll 1
                for (unsigned r = 0; r < rows; ++r) {
                    bulk(to + r * e.z, base + static_cast<size_t>(e.x) * 16u + r * stride, e.z, bar, once);
                    if (two) bulk(to + part + r * e.z, base + static_cast<size_t>(e.y) * 16u + r * stride, e.z, bar, once);
                }
            }
            return true;
        },
        [&](const unsigned char *k, const unsigned char *v, int n, unsigned bytes) {
            const int row_bytes = p.D * (Q8 ? 1 : 2);
            const KvBlock b(n, row_bytes);
            unsigned bar;
            const unsigned to = room(2u * bytes, static_cast<unsigned>(b.bytes()), bar);
            if (!ok) return false;
            bulk(to, k, bytes, bar, keep);
#pragma unroll 1
            for (int i = 0; i * b.R < n; ++i)
                bulk(to + b.v_at + i * b.v_stride, v + static_cast<size_t>(i * b.R) * row_bytes, static_cast<unsigned>(min(b.R, n - i * b.R) * row_bytes), bar, keep);
            return true;
        });
    drain(sh.full, ST_BARS, issued);
}
// ... another asks L2 for what comes after it, at most prefetch_bytes ahead: the ring alone holds too little to keep HBM busy
// through the exchanges, and a refill from L2 comes at more than twice the rate of HBM.
template <bool Q8, int MT>
__device__ __forceinline__ void feed_l2(Ctx<MT> &c) {
    Shared<MT> &sh = c.sh();
    const StepParams &p = c.p();
    const unsigned ahead = static_cast<unsigned>(p.prefetch_bytes) >> 4;
    if (ahead == 0) return;
    const unsigned char *const lm_map = p.maps + static_cast<size_t>(4 * p.n_layers) * 128;
    unsigned pos = 0;
    bool ok = true;
    auto due = [&](unsigned bytes) {             // waits until the chunk is near enough; false: the ring has it already (or gave up)
        pos += bytes >> 4;
        unsigned spins = 0;
        int lead;                                // (differences: the counters may wrap)
        while ((lead = static_cast<int>(pos - *reinterpret_cast<volatile unsigned *>(&sh.sent))) > static_cast<int>(ahead)) {
            if (*c.abort() || ++spins > (1u << 22)) { ok = false; return false; }      // bounded; a hint not given costs only time
            __nanosleep(64);
        }
        return lead > 0;
    };
    auto ask = [&](const unsigned char *from, unsigned bytes) { asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(from), "r"(bytes) : "memory"); };
    for_each_chunk<Q8>(
        c,
        [&](const unsigned char *base, const uint4 &e, const unsigned char *map) {
            const bool two = e.y != ~0u;
            const unsigned rows = e.w >> 16, part = e.z * (rows == 0u || rows == ST_BOX ? 1u : rows);
            if (!due(two ? 2u * part : part)) return ok;
            if (rows == 0u) {
                ask(base + static_cast<size_t>(e.x) * 16u, part);
                if (two) ask(base + static_cast<size_t>(e.y) * 16u, part);
            } else if (rows == ST_BOX && p.map_fence != 2 && map != lm_map) {          // (only through maps that are never rewritten)
                asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(0), "r"(e.x), "r"(e.w & 0xffffu) : "memory");
                if (two) asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(0), "r"(e.y), "r"(e.w & 0xffffu) : "memory");
            }
            return true;
        },
        [&](const unsigned char *k, const unsigned char *v, int, unsigned bytes) {
            if (!due(2u * bytes)) return ok;
            ask(k, bytes);
            ask(v, bytes);
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
    const int tiles = (sh.u1[ST_DN] - sh.u0[ST_DN] + p.cols[ST_DN].tile - 1) / p.cols[ST_DN].tile;
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
    drain(sh.x_full, 4u, k);
}

}  // namespace ST_NS
}  // namespace edgefm
