// Parameters and launch layout of the persistent decode-step kernel (step_kernel.cuh).
#pragma once
#include <algorithm>
#include <cmath>
#include <cstring>

#include "../../include/edgefm.h"
#include "common.cuh"
#include "tensor_map.h"

namespace edgefm {

constexpr int ST_NW = 8;                     // consumer warps per CTA
constexpr int ST_NT = ST_NW * 32;
constexpr int ST_THREADS = ST_NT + 128;      // + the feeding warpgroup (two of its warps work)
// Registers: 384 threads are launched with 168 each; 256 x 208 + 128 x 88 is what they were launched with.
constexpr int ST_REGS_LAUNCH = 168, ST_REGS = 208, ST_REGS_FEED = 88;
static_assert(ST_NT * ST_REGS + 128 * ST_REGS_FEED <= ST_THREADS * ST_REGS_LAUNCH, "setmaxnreg only redistributes the launch's registers");
constexpr unsigned ST_DRAIN_NS = 2000000000u;   // how long a CTA that leaves waits for its copies in flight
constexpr int ST_BARS = 16;                  // chunks the ring can hold at once (a power of two)
constexpr int ST_CHUNK_BYTES = 52 * 1024;    // aimed at for a ring chunk cut by columns
constexpr int ST_CHUNK_SMALL = 28 * 1024;    // ... where a segment needs no exchange of its own: the ring refills in finer steps (1.5B shape, 8960 columns: 6.0 -> 5.5 us)
constexpr int ST_ACT_WHOLE = 72 * 1024;      // MLP activations up to this size are staged whole
constexpr int ST_CHUNK_WHOLE = 68 * 1024;    // a tile of whole rows may be this large
constexpr int ST_TILE = 16;                  // rows of a tile: the M of one m16n8k16 tensor-core instruction (pairs: 8 and their partners)
// cached positions per ring chunk: a warp multiplies 16 of them by 64 dims
__host__ __device__ constexpr int kv_block(int D) { return 16 * ST_NW / (D / 64); }
constexpr int ST_MIN_CHUNK = 16;             // fewest cached positions a CTA attends to (shorter contexts occupy fewer CTAs)
constexpr int ST_PREFETCH_BYTES = 256 * 1024;   // L2 look-ahead per CTA beyond the ring (160 KB: 1.5B shape + 1 %; 352 KB: 7B shape + 1 %)
constexpr int ST_KEEP = 4;                   // 64-column blocks of the input vector a warp can keep in registers with tiles of 16 rows ...
constexpr int ST_KEEP_HALF = 8;              // ... and of 8

// Tokens a call may carry (a build of the kernel each): 1, 2, 4 or 8.  bf16 pieces an activation value is multiplied as: three (24 mantissa
// bits) for one or two tokens, two (16 bits, twice the precision of the weights) for more; the pieces of all tokens are columns
// of the tensor-core instruction's B operand, 8 per instruction.
__host__ __device__ constexpr int st_pieces(int mt) { return mt <= 2 ? 3 : 2; }
__host__ __device__ constexpr int st_arrays(int mt) { return mt * st_pieces(mt); }
// How vectors are exchanged (step_kernel.cuh): polled packets, or written plainly and fetched after an arrival.
__host__ __device__ constexpr bool st_packets(int mt) { return mt <= 2; }
// rows whose partial sums meet in shared memory at a time
__host__ __device__ constexpr int st_batch(int mt) { return mt <= 2 ? 128 : mt == 4 ? 64 : 32; }

enum { ST_QKV = 0, ST_O = 1, ST_GU = 2, ST_DN = 3, ST_LM = 4 };

// How an operator with rows of K values is cut: tiles of 16 rows (8 pairs), or of 8 rows (4 pairs) where 16 whole ones are too long for a
// ring chunk (half of the MMA idles, but chunks stay contiguous and the input vector in registers: K = 3584, gate/up 5.9 TB/s by
// segments and 6.6 so); a tile whose rows are longer still is cut into `segs` segments of `seg` columns.  All warps work on every chunk: warp w multiplies the 64-column blocks [nb w / 8, nb (w + 1) / 8) of
// the nb blocks of the chunk, and so needs only that part of the input vector.
// A segment comes as one box (two for pairs) of a tensor map: box_rows rows (what lies past the tile is fetched and not used, so a
// CTA's rows are dealt out evenly to its tiles: 25 rows as 13 + 12, not 16 + 9) x seg columns, delivered as [64-column block][row][128 bytes].  (One bulk copy per row segment costs the copy unit about
// 150 cycles whatever its size: 11 rows of 4 KB took 2.6 TB/s, as a box they come at the rate of whole rows.)  box_rows 0: K is not a
// multiple of 64, one copy per row segment.
struct StepCols {
    int K, seg, segs, box_rows;
    int tile;            // units (rows or pairs) of a tile
};

// Pointers of a layer; entry [n_layers] describes the output layer.
struct StepLayer {
    const uint16_t *wqkv, *wo, *w_gate_up, *w_down;
    const uint16_t *input_norm, *post_norm, *bqkv;
    long long pad_;
};
struct StepHead {
    const uint16_t *lm_head, *final_norm;
    int rows, remap;     // remap: row r stands for token vocab_ids[r] (a pruned vocabulary)
    long long pad_[5];
};
static_assert(sizeof(StepLayer) == 64 && sizeof(StepHead) == 64, "one table of 64-byte entries");

struct StepParams {
    int n_layers, H, nq, nkv, G, D, F, V;
    int qd;                        // nq * D
    int half_shift;                // log2(D / 2)
    float eps, q_scale;            // q_scale: 1 / sqrt(D) * log2(e) (the softmax works in powers of two)
    int max_context;
    uint16_t *k_cache, *v_cache;   // [L][nkv][max_context][D] bf16, or signed bytes (compressed cache)
    float *k_scale, *v_scale;      // compressed cache: [L][nkv][max_context]
    const uint16_t *embed;
    const double *inv_freq;        // [D / 2]
    const StepLayer *layers;       // [n_layers + 1]
    const unsigned char *maps;     // CUtensorMap [4 n_layers + 1] of the operators that are cut into boxes (128 bytes each)
    int map_fence;                 // maps the host may have rewritten since the last launch: 1 the output layer's, 2 all
    const int *vocab_ids;
    StepState *state;
    StepRequest req;
    // Vectors that are multiplied next: as they lie in shared memory, arrays of bf16 pieces [token * S + piece][st_array_bytes(K)], zero past
    // K; behind the residual streams' arrays the CTAs' sums of squares [token][ss_stride].  act: [segment][array][st_array_bytes(seg)].
    unsigned char *x_vec;          // residual stream after the down projection, times the next norm's weight
    unsigned char *xo_vec;         // ... after the O projection
    unsigned char *ao_vec;         // attention output
    unsigned char *act_vec;        // MLP activations
    int ss_stride;
    unsigned *arrivals;            // CTAs that have written their share, all exchanges of all calls
    // One or two tokens: the same vectors as packets of 8 bytes, {three bf16 pieces, 16-bit tag}, [token] first
    unsigned long long *x_ll, *xo_ll;   // per CTA one line of x_line packets, its last one the CTA's sum of squares {fp32, 32-bit tag}
    unsigned long long *ao_ll;     // per CTA one line of ao_line packets
    unsigned long long *act_ll;    // [act_len]
    int x_line, ao_line, act_len;
    int act_packets;               // 1: the MLP activations are staged whole, from packets; 0: they come by segments
    // packets of 8 bytes {fp32 value, tag}
    unsigned long long *q_ll;      // rotated q, k and v: [token], per CTA one line of q_line packets, {lo, hi} of its row pairs in order
    unsigned long long *part_ll;   // attention partial results [token and chunk][nq D] (unnormalised)
    unsigned long long *stat_ll;   // ... their {maximum, denominator} [token and chunk][nq][2]
    unsigned long long *lm_ll;     // greedy candidates: per CTA one line, {value, row} of every token
    int q_line;
    StepCols cols[5];              // per operator
    int ring_bytes, list_at, resid_at, table_bytes;   // shared memory (list_at, resid_at: inside the tables)
    int act_slots;                 // segments of the MLP activations in shared memory
    int prefetch_bytes;            // how far the L2 prefetch runs ahead of the ring
    int epoch_slot;                // which of the state's epochs tags this build's packets
    int barrier_extra;             // test hook: an exchange waits for one arrival more than there are CTAs (1; 0 in production)
    unsigned spin_limit;           // upper bound of every device-side wait, nanoseconds
    unsigned long long *prof;      // optional timestamps [gridDim.x][prof_stride]
    int prof_stride;
    // tight builds only
    int kv_block;                  // cached positions per ring chunk
    const unsigned *unit_tab;      // unit tables of the lines (residual stream, attention output)
    int merged_at, merged_len;     // attention outputs of this CTA: inside the tables; at most per token
};

using StepKernel = void (*)(const StepParams);
// one kernel per head size, query heads per kv head, cache format, tokens per call and room in shared memory (null: not built)
StepKernel step_kernel_for(int D, int G, bool kv8, int mt, bool tight);
// First unit (of n) of CTA c (n * ncta below 2^32: checked by step_plan; a 64-bit division would cost the feeding thread more than a copy).
__host__ __device__ inline int st_first(int n, int c, int ncta) { return static_cast<int>(static_cast<unsigned>(n) * static_cast<unsigned>(c) / static_cast<unsigned>(ncta)); }
__host__ __device__ inline int st_line(int most) { return (most + 15) / 16 * 16; }   // packets of a line: whole 128 bytes

// How an operator with rows of K values is cut of which a CTA owns at most `most` units (rows, or pairs).
inline StepCols step_cols(int K, int most, bool paired, int max_seg, int chunk_bytes, int chunk_whole) {
    const int full = paired ? ST_TILE / 2 : ST_TILE, per_unit = paired ? 4 * K : 2 * K;     // bytes
    StepCols c{K, K, 1, 0, full};
    if (K <= max_seg && std::min(most, full) * per_unit <= chunk_whole) return c;
    c.tile = full / 2;
    if (K <= max_seg && c.tile * per_unit <= chunk_whole && K <= ST_KEEP_HALF * ST_NW * 64) return c;
    const int tiles = (most + full - 1) / full;
    c.tile = (most + tiles - 1) / tiles;
    const int rows = paired ? 2 * c.tile : c.tile;
    const int cols = std::min(max_seg, std::max(512, chunk_bytes / (2 * rows) / 512 * 512));
    const int n = (K + cols - 1) / cols;
    c.seg = std::min(cols, ((K + n - 1) / n + 511) / 512 * 512);      // a whole number of blocks for every warp
    c.segs = (K + c.seg - 1) / c.seg;
    if (K % 64 == 0) c.box_rows = c.tile;
    return c;
}
// Bytes between the arrays of a staged vector of n columns: whole 64-column blocks, + 64 so that neighbouring arrays use other banks.
__host__ __device__ inline int st_array_bytes(int n) { return (n + 63) / 64 * 128 + 64; }

// ---- launch plan (host) ------------------------------------------------------------------------------------------------
struct StepLaunch {
    StepKernel kernel = nullptr;
    StepParams p{};
    int grid = 0;
    size_t dyn_smem = 0;
    size_t ll_bytes = 0;        // exchange buffers (zeroed once: tag 0 is never used, columns past K stay zero), then the unit tables of a tight build
    size_t unit_tab_bytes = 0;  // unit tables in global memory (0: in shared memory)
    int max_chunk_bytes = 0;
    int list_len = 0;           // chunks the list in shared memory has room for
};
int step_shared_bytes(int mt);  // fixed part of the kernel's shared memory
int step_scratch_floats(int D, int G, int mt);
// The chunks CTA `cta` streams of an operator, six words each: the entry (chunk_entry), first unit, units.  Returns how many there are.
int step_chunks(const StepLaunch &sl, int op, int cta, unsigned *out, int capacity);

// Packets of the attention's maxima and denominators; whole lines (what follows is lines with one writer each: 64 bytes off, two share one).
inline size_t step_stat_len(size_t chunks, int nq) { return (chunks * nq * 2 + 15) / 16 * 16; }
// Bytes of a vector's exchange buffer / of the MLP activations' (whole 128 bytes).
inline size_t step_vec_bytes(const StepParams &p, int mt, int K, bool sums) {
    return (static_cast<size_t>(st_arrays(mt)) * st_array_bytes(K) + (sums ? 4 * static_cast<size_t>(mt) * p.ss_stride : 0) + 127) / 128 * 128;
}
inline size_t step_act_bytes(const StepParams &p, int mt) {
    return (static_cast<size_t>(p.cols[ST_DN].segs) * st_arrays(mt) * st_array_bytes(p.cols[ST_DN].seg) + 127) / 128 * 128;
}
// What a plan asks of the shared memory.  The first form suits every shape in use.  The tight ones give up speed for room where a CTA owns more than
// 128 attention outputs, or vectors, rows or the vocabulary are so long that it does not fit: tables and chunk list out of shared
// memory, then smaller chunks, then fewer cached positions per chunk.
struct StepRoom { bool tight; int chunk_bytes, chunk_small, chunk_whole, kv_share; };
constexpr StepRoom ST_ROOM[] = {{false, ST_CHUNK_BYTES, ST_CHUNK_SMALL, ST_CHUNK_WHOLE, 1}, {true, ST_CHUNK_BYTES, ST_CHUNK_SMALL, ST_CHUNK_WHOLE, 1},
                                {true, 32 * 1024, ST_CHUNK_SMALL, 32 * 1024, 1}, {true, 16 * 1024, 16 * 1024, 16 * 1024, 2}};
constexpr int ST_TIGHT_ROW_BITS = 15;     // row of an entry of the tight builds' unit tables

// Shared-memory split and exchange buffers for a model shape.  Returns null, or why the shape does not fit.
inline const char *step_plan_in(const StepRoom &room, const edgefm_shape &sh, int max_context, int num_sms, int smem_optin, bool kv8, int mt, StepLaunch *sl) {
    const int H = sh.hidden, D = sh.head_dim, nq = sh.n_q_heads, nkv = sh.n_kv_heads, F = sh.ffn, qd = nq * D, G = nq / nkv;
    StepParams &p = sl->p;
    sl->kernel = step_kernel_for(D, G, kv8, mt, room.tight);
    if (!sl->kernel) return "no step kernel for this combination of options";
    // every CTA must own a row of the residual stream: its contribution is what says that it has read the exchange before
    const int grid = sl->grid = std::min(num_sms, H);
    const long long units = std::max({static_cast<long long>(sh.vocab), static_cast<long long>(F), static_cast<long long>(nq + 2 * nkv) * D / 2, static_cast<long long>(max_context)});
    if ((!room.tight && qd > 128 * grid) || (units + 1) * (grid + 1) > 0x7fffffffLL) return "model shape does not fit the step kernel";
    p.n_layers = sh.n_layers; p.H = H; p.nq = nq; p.nkv = nkv; p.G = G; p.D = D; p.F = F; p.V = sh.vocab; p.qd = qd;
    p.half_shift = D == 64 ? 5 : 6;
    p.eps = sh.rms_eps;
    p.q_scale = static_cast<float>(1.4426950408889634 / std::sqrt(static_cast<double>(D)));
    p.max_context = max_context;
    auto most = [&](int n) { return (n + grid - 1) / grid; };
    const int q_most = most((nq + 2 * nkv) * D / 2);
    p.cols[ST_QKV] = step_cols(H, q_most, true, 1 << 30, room.chunk_bytes, room.chunk_whole);
    p.cols[ST_GU] = step_cols(H, most(F), true, 1 << 30, room.chunk_bytes, room.chunk_whole);
    p.cols[ST_LM] = step_cols(H, most(sh.vocab), false, 1 << 30, room.chunk_bytes, room.chunk_whole);
    p.cols[ST_O] = step_cols(qd, most(H), false, 1 << 30, room.chunk_bytes, room.chunk_whole);
    // the activations whole if they leave the ring room to cover the latency of HBM (7B: 113 KB for them, and the stream fell to 3.9 TB/s)
    p.act_packets = st_packets(mt) && st_arrays(mt) * st_array_bytes(F) <= ST_ACT_WHOLE;
    p.cols[ST_DN] = step_cols(F, most(H), false, mt <= 2 ? 2048 : 1024,       // (two segments of activations are in shared memory, as pieces)
                              p.act_packets ? room.chunk_small : room.chunk_bytes, room.chunk_whole);
    // (a chunk's place is counted in 16-byte units of its matrix, 32 bits of them; boxes are placed by rows)
    const long long rows_of[5] = {static_cast<long long>(nq + 2 * nkv) * D, H, 2LL * F, H, sh.vocab};
    for (int o = 0; o < 5; ++o)
        if (p.cols[o].box_rows == 0 && rows_of[o] * (p.cols[o].K / 8) > 0xffffffffLL) return "a weight matrix is larger than 64 GiB";
    p.q_line = st_line(2 * most((nq + 2 * nkv) * D / 2));
    p.ss_stride = (grid + 3) / 4 * 4;
    p.x_line = st_line(most(H) + 1);
    p.ao_line = st_line(2 * most(qd / 2));
    p.act_len = (F + 15) / 16 * 16;
    const int total_x = grid * ((most(H) + 1) / 2), total_a = grid * most(qd / 2), row_bits = room.tight ? ST_TIGHT_ROW_BITS : 16, rows = 1 << row_bits, lines = 1 << (30 - row_bits);
    if (st_packets(mt) && (H >= rows || qd >= rows || grid * p.x_line / 2 >= lines || grid * p.ao_line / 2 >= lines)) return "model shape does not fit the step kernel";
    const int unit_bytes = st_packets(mt) ? 4 * (total_x + total_a) : 0;
    sl->unit_tab_bytes = room.tight ? unit_bytes : 0;
    p.list_at = ((sh.n_layers + 1) * 64 + (room.tight ? 0 : unit_bytes) + 15) / 16 * 16;
    // the chunk list: tiles of the busiest CTA (QKV tiles are also cut at the ends of head halves) x segments
    auto listed = [&](int op, int n) { return (most(n) + p.cols[op].tile - 1) / p.cols[op].tile * p.cols[op].segs; };
    const int chunks_listed = (q_most / p.cols[ST_QKV].tile + 2 * (q_most / (D / 2) + 2)) * p.cols[ST_QKV].segs + listed(ST_O, H) + listed(ST_DN, H) + listed(ST_GU, F) + listed(ST_LM, sh.vocab);
    sl->list_len = room.tight ? 0 : chunks_listed;
    p.merged_at = p.list_at + 16 * sl->list_len;
    p.merged_len = 2 * most(qd / 2);
    p.resid_at = p.merged_at + (room.tight ? 4 * mt * p.merged_len : 0);
    p.table_bytes = (p.resid_at + 4 * mt * most(H) + 127) / 128 * 128;
    // one area for the staged vector, the attention's scratch and the segments of the MLP activations: they follow one another
    const int slot = st_arrays(mt) * st_array_bytes(p.cols[ST_DN].seg), vec = std::max(st_arrays(mt) * st_array_bytes(H) + 4 * mt * p.ss_stride, st_arrays(mt) * st_array_bytes(qd));
    int area = std::max(vec, 4 * step_scratch_floats(D, G, mt));
    p.act_slots = p.cols[ST_DN].segs == 1 ? 1 : std::max(mt == 4 ? 3 : 2, std::min(3, area / slot));     // (every slot is taken from the ring)
    area = std::max(area, p.act_packets ? st_arrays(mt) * st_array_bytes(F) : p.act_slots * slot);
    const int fixed = step_shared_bytes(mt) + p.table_bytes + (area + 127) / 128 * 128;
    p.kv_block = kv_block(D) / room.kv_share;
    int chunk = p.kv_block * D * (kv8 ? 2 : 4) + 4 * 32;      // (K rows, then V in four quarters 32 bytes apart)
    const int owned[5] = {q_most, most(H), most(F), most(H), most(sh.vocab)};
    for (int o = 0; o < 5; ++o) chunk = std::max(chunk, std::min(owned[o], p.cols[o].tile) * (o == ST_QKV || o == ST_GU ? 4 : 2) * p.cols[o].seg);
    sl->max_chunk_bytes = (chunk + 127) / 128 * 128;
    const int ring = (smem_optin - fixed) / 128 * 128;
    if (ring < sl->max_chunk_bytes) return "model shape does not fit the shared memory";
    p.ring_bytes = ring;
    sl->dyn_smem = static_cast<size_t>(fixed) + ring;
    p.prefetch_bytes = ST_PREFETCH_BYTES;
    p.spin_limit = 1000000000u;   // 1 s
    const size_t chunks = static_cast<size_t>(std::max(grid / nkv, mt));
    sl->ll_bytes = 8 * (static_cast<size_t>(grid) * mt * p.q_line + static_cast<size_t>(grid) * 16 + chunks * qd + step_stat_len(chunks, nq)) + 2 * step_vec_bytes(p, mt, H, true) +
                   step_vec_bytes(p, mt, qd, false) + step_act_bytes(p, mt) + 256 +
                   (st_packets(mt) ? 8 * (static_cast<size_t>(grid) * mt * (2 * p.x_line + p.ao_line) + static_cast<size_t>(mt) * p.act_len) : 0) + (sl->unit_tab_bytes + 255) / 256 * 256;
    return nullptr;
}
inline const char *step_plan(const edgefm_shape &sh, int max_context, int num_sms, int smem_optin, bool kv8, int mt, StepLaunch *sl) {
    const char *why = nullptr;
    for (const StepRoom &room : ST_ROOM) {
        if (!(why = step_plan_in(room, sh, max_context, num_sms, smem_optin, kv8, mt, sl))) return nullptr;
        if (mt == 8) break;      // (the prompt kernels verify such a block)
    }
    return why;
}
// The unit tables of a tight build, as the others make them in shared memory (make_table).
inline void step_unit_table(const StepLaunch &sl, unsigned *tab) {
    const StepParams &p = sl.p;
    for (int v = 0; v < 2; ++v) {
        const int n = v ? p.qd : p.H, grain = v ? 2 : 1, line = v ? p.ao_line : p.x_line, upl = ((n / grain + sl.grid - 1) / sl.grid * grain + 1) / 2;
        for (int w = 0; w < sl.grid; ++w) {
            int row = st_first(n / grain, w, sl.grid) * grain;
            const int r1 = st_first(n / grain, w + 1, sl.grid) * grain;
            for (int e = 0; e < upl; ++e, row += 2)
                *tab++ = static_cast<unsigned>(row & ((1 << ST_TIGHT_ROW_BITS) - 1)) | static_cast<unsigned>(std::max(0, std::min(2, r1 - row))) << ST_TIGHT_ROW_BITS |
                         static_cast<unsigned>(w * (line >> 1) + e) << (ST_TIGHT_ROW_BITS + 2);
        }
    }
}
// Wire the exchange buffers (256-byte aligned base).
inline void step_wire(StepLaunch *sl, int mt, unsigned long long *base) {
    StepParams &p = sl->p;
    const size_t g = static_cast<size_t>(sl->grid), m = static_cast<size_t>(mt), chunks = static_cast<size_t>(std::max(sl->grid / p.nkv, mt));
    unsigned char *b = reinterpret_cast<unsigned char *>(base);
    p.arrivals = reinterpret_cast<unsigned *>(b); b += 256;
    p.x_vec = b; b += step_vec_bytes(p, mt, p.H, true);
    p.xo_vec = b; b += step_vec_bytes(p, mt, p.H, true);
    p.ao_vec = b; b += step_vec_bytes(p, mt, p.qd, false);
    p.act_vec = b; b += step_act_bytes(p, mt);
    base = reinterpret_cast<unsigned long long *>(b);
    p.q_ll = base; base += g * m * p.q_line;
    p.lm_ll = base; base += g * 16;
    p.part_ll = base; base += chunks * p.qd;
    p.stat_ll = base; base += step_stat_len(chunks, p.nq);
    if (!st_packets(mt)) return;
    p.x_ll = base; base += g * m * p.x_line;
    p.xo_ll = base; base += g * m * p.x_line;
    p.ao_ll = base; base += g * m * p.ao_line;
    p.act_ll = base; base += m * p.act_len;
    p.unit_tab = sl->unit_tab_bytes ? reinterpret_cast<const unsigned *>(base) : nullptr;
}
// Tensor map of a row-major bf16 [rows][K] matrix for the boxes of an operator: the 64-column blocks of a row are the last dimension.
inline bool step_map(CUtensorMap *m, const StepCols &c, const void *base, int rows) {
    std::memset(m, 0, sizeof *m);
    if (c.box_rows == 0) return true;
    TensorMapEncodeFn enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[3] = {64, static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(c.K / 64)}, strides[2] = {static_cast<cuuint64_t>(c.K) * 2, 128};
    const cuuint32_t box[3] = {64, static_cast<cuuint32_t>(c.box_rows), static_cast<cuuint32_t>(c.seg / 64)}, es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// All of them: [4 layer + operator], the output layer last.
inline bool step_maps(const StepParams &p, const edgefm_layer_weights *layers, const void *lm_head, int lm_rows, CUtensorMap *maps) {
    for (int l = 0; l < p.n_layers; ++l) {
        const edgefm_layer_weights &w = layers[l];
        if (!step_map(maps + 4 * l + ST_QKV, p.cols[ST_QKV], w.wqkv, (p.nq + 2 * p.nkv) * p.D) || !step_map(maps + 4 * l + ST_O, p.cols[ST_O], w.wo, p.H) ||
            !step_map(maps + 4 * l + ST_GU, p.cols[ST_GU], w.w_gate_up, 2 * p.F) || !step_map(maps + 4 * l + ST_DN, p.cols[ST_DN], w.w_down, p.H))
            return false;
    }
    return step_map(maps + 4 * p.n_layers, p.cols[ST_LM], lm_head, lm_rows);
}
// One entry per layer, then the output layer.
inline void step_layers(const edgefm_shape &sh, const edgefm_layer_weights *layers, const void *final_norm, const void *lm_head, StepLayer *out) {
    auto u16 = [](const void *q) { return static_cast<const uint16_t *>(q); };
    for (int l = 0; l < sh.n_layers; ++l) {
        const edgefm_layer_weights &w = layers[l];
        out[l] = StepLayer{u16(w.wqkv), u16(w.wo), u16(w.w_gate_up), u16(w.w_down), u16(w.input_norm), u16(w.post_norm), sh.qkv_bias ? u16(w.bqkv) : nullptr, 0};
    }
    StepHead h{u16(lm_head), u16(final_norm), sh.vocab, 0, {}};
    std::memcpy(&out[sh.n_layers], &h, sizeof h);
}

}  // namespace edgefm
