// Parameters and launch layout of the persistent decode-step kernel (step_kernel.cuh).
#pragma once
#include <algorithm>
#include <cmath>
#include <cstring>

#include "../../include/edgefm.h"
#include "common.cuh"

namespace edgefm {

constexpr int ST_NW = 8;                     // consumer warps per CTA
constexpr int ST_NT = ST_NW * 32;
constexpr int ST_THREADS = ST_NT + 128;      // + the feeding warpgroup (two of its warps work)
// Registers: 384 threads are launched with 168 each; 256 x 216 + 128 x 72 is what they were launched with.
constexpr int ST_REGS_LAUNCH = 168, ST_REGS = 216, ST_REGS_FEED = 72;
static_assert(ST_NT * ST_REGS + 128 * ST_REGS_FEED <= ST_THREADS * ST_REGS_LAUNCH, "setmaxnreg only redistributes the launch's registers");
constexpr int ST_BARS = 16;                  // chunks the ring can hold at once (a power of two)
constexpr int ST_CHUNK_BYTES = 52 * 1024;    // at most, for a ring chunk of more than one row (or pair)
constexpr int ST_BATCH = 64;                 // output units whose partial sums meet in shared memory at a time (pairs: two rows each)
constexpr int ST_KV_BLOCK = 8 * ST_NW;       // cached positions per ring chunk: eight per warp
constexpr int ST_MIN_CHUNK = 16;             // fewest cached positions a CTA attends to (shorter contexts occupy fewer CTAs)
#ifndef ST_PREFETCH_VALUE
#define ST_PREFETCH_VALUE (352 * 1024)
#endif
constexpr int ST_PREFETCH_BYTES = ST_PREFETCH_VALUE;   // L2 look-ahead per CTA beyond the ring

enum { ST_QKV = 0, ST_O = 1, ST_GU = 2, ST_DN = 3, ST_LM = 4 };

// How the columns of a row are dealt out: warp w takes the 16-byte pieces (8 columns) [K8 w / 8, K8 (w + 1) / 8) of EVERY row of its
// CTA.  Inside a warp a row is read by `1 << lpr_log2` neighbouring lanes, `pieces` pieces each; 32 >> lpr_log2 rows at a time.
struct StepCols {
    int K, K8;
    int lpr_log2;        // 3, 4 or 5
    int pieces;
    int variant;         // ST_V*: pieces a lane multiplies at once (and keeps in registers if there are no more), row groups folded together
    int rows_per_chunk;  // rows of a ring chunk
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
    const int *vocab_ids;
    StepState *state;
    const StepRequest *req;
    // exchange buffers: packets {value, tag}, 8 bytes each
    unsigned long long *x_ll;      // residual stream after the down projection: per CTA one line of x_line packets
    unsigned long long *xo_ll;     // ... after the O projection
    unsigned long long *q_ll;      // rotated q, k and v: per CTA one line of q_line packets, {lo, hi} of its row pairs in order
    unsigned long long *ao_ll;     // attention output: per CTA one line of ao_line packets
    unsigned long long *act_ll;    // MLP activations [F]
    unsigned long long *part_ll;   // attention partial results [chunks][nq D] (unnormalised)
    unsigned long long *stat_ll;   // ... their {maximum, denominator} [chunks][nq][2]
    unsigned long long *lm_ll;     // greedy candidates: per CTA one line of 16 packets {value, row}
    int x_line, q_line, ao_line;
    StepCols cols[5];              // per operator
    int ring_bytes, resid_at, table_bytes, xs_floats;   // shared memory (resid_at: inside the tables)
    int prefetch_bytes;            // how far the L2 prefetch runs ahead of the ring
    int barrier_extra;             // test hook: 1 = the packets expected never come, so that the first wait runs out
    unsigned spin_limit;           // upper bound of every device-side wait, nanoseconds
    unsigned long long *prof;      // optional timestamps [gridDim.x][prof_stride]
    int prof_stride;
};

using StepKernel = void (*)(const StepParams);
// one kernel per head size, query heads per kv head and cache format
StepKernel step_kernel_d64(int G);
StepKernel step_kernel_d128(int G);
StepKernel step_kernel_q8_d64(int G);
StepKernel step_kernel_q8_d128(int G);

// First unit (of n) of CTA c (n * ncta below 2^32: checked by step_plan; a 64-bit division would cost the feeding thread more than a copy).
__host__ __device__ inline int st_first(int n, int c, int ncta) { return static_cast<int>(static_cast<unsigned>(n) * static_cast<unsigned>(c) / static_cast<unsigned>(ncta)); }
__host__ __device__ inline int st_line(int most) { return (most + 15) / 16 * 16; }   // packets of a line: whole 128 bytes

// Variants of the products: ST_V<pieces><row groups>.  Short rows are multiplied 4 groups at a time (more independent sums, fewer
// folds), long ones two or one, since a chunk holds few of them.
enum { ST_V14 = 0, ST_V24 = 1, ST_V34 = 2, ST_V52 = 3, ST_V62 = 4, ST_V101 = 5, ST_N_VARIANTS = 6 };
constexpr int ST_VARIANTS[ST_N_VARIANTS][2] = {{1, 4}, {2, 4}, {3, 4}, {5, 2}, {6, 2}, {10, 1}};
// Columns of an operator with rows of K values.  paired: its units are two rows.
inline StepCols step_cols(int K, bool paired) {
    StepCols c{};
    c.K = K;
    c.K8 = K / 8;
    const int most = (c.K8 + ST_NW - 1) / ST_NW, fit = std::max(1, ST_CHUNK_BYTES / (2 * K));   // pieces of the busiest warp; rows of a chunk
    // least work: lanes x pieces, padded to whole groups; more if the vector does not stay in registers and is re-read for every group
    // of rows; per-group overhead
    double best = 1e9;
    for (int lg = 5; lg >= 3; --lg)
        for (int v = 0; v < ST_N_VARIANTS; ++v) {
            const int pg = ST_VARIANTS[v][0], group = (32 >> lg) * ST_VARIANTS[v][1];
            const int pieces = (most + (1 << lg) - 1) >> lg, slots = (pieces + pg - 1) / pg * pg;
            if (group > fit && !(lg == 5 && v == ST_V101)) continue;
            double cost = (slots << lg) * (pieces <= pg ? 1.0 : 1.3) * (1.0 + 0.01 * lg);
            cost *= 1.0 + 0.15 / ST_VARIANTS[v][1];
            if (cost < best) { best = cost; c.lpr_log2 = lg; c.pieces = pieces; c.variant = v; }
        }
    const int group = (32 >> c.lpr_log2) * ST_VARIANTS[c.variant][1];
    c.rows_per_chunk = std::max(fit / group * group, std::min(group, fit));
    if (paired) c.rows_per_chunk = std::max(2, c.rows_per_chunk / 2 * 2);
    return c;
}

// ---- launch plan (host) ------------------------------------------------------------------------------------------------
struct StepLaunch {
    StepKernel kernel = nullptr;
    StepParams p{};
    int grid = 0;
    size_t dyn_smem = 0;
    size_t ll_bytes = 0;        // exchange buffers (zeroed once: tag 0 is never used)
    int max_chunk_bytes = 0;
};
int step_shared_bytes();        // fixed part of the kernel's shared memory
int step_scratch_floats(int D, int G);

// Shared-memory split and exchange buffers for a model shape.  Returns null, or why the shape does not fit.
inline const char *step_plan(const edgefm_shape &sh, int max_context, int num_sms, int smem_optin, bool kv8, StepLaunch *sl) {
    const int H = sh.hidden, D = sh.head_dim, nq = sh.n_q_heads, nkv = sh.n_kv_heads, F = sh.ffn, qd = nq * D, G = nq / nkv;
    StepParams &p = sl->p;
    sl->kernel = D == 64 ? (kv8 ? step_kernel_q8_d64(G) : step_kernel_d64(G)) : (kv8 ? step_kernel_q8_d128(G) : step_kernel_d128(G));
    // every CTA must own a row of the residual stream: its contribution is what says that it has read the exchange before
    const int grid = sl->grid = std::min(num_sms, H);
    const long long units = std::max({static_cast<long long>(sh.vocab), static_cast<long long>(F), static_cast<long long>(nq + 2 * nkv) * D / 2, static_cast<long long>(max_context)});
    if (nkv > grid || qd > 2 * ST_NT * grid || H >= 65536 || qd >= 65536 || (units + 1) * (grid + 1) > 0x7fffffffLL) return "model shape does not fit the step kernel";
    p.n_layers = sh.n_layers; p.H = H; p.nq = nq; p.nkv = nkv; p.G = G; p.D = D; p.F = F; p.V = sh.vocab; p.qd = qd;
    p.half_shift = D == 64 ? 5 : 6;
    p.eps = sh.rms_eps;
    p.q_scale = static_cast<float>(1.4426950408889634 / std::sqrt(static_cast<double>(D)));
    p.max_context = max_context;
    p.cols[ST_QKV] = step_cols(H, true); p.cols[ST_O] = step_cols(qd, false); p.cols[ST_GU] = step_cols(H, true);
    p.cols[ST_DN] = step_cols(F, false); p.cols[ST_LM] = step_cols(H, false);
    auto most = [&](int n) { return (n + grid - 1) / grid; };
    p.x_line = st_line(most(H));
    p.q_line = st_line(2 * most((nq + 2 * nkv) * D / 2));
    p.ao_line = st_line(2 * most(qd / 2));
    const int total_x = grid * ((most(H) + 1) / 2), total_a = grid * most(qd / 2);
    if (grid * p.x_line / 2 >= 16384 || grid * p.ao_line / 2 >= 16384) return "model shape does not fit the step kernel";
    p.resid_at = (sh.n_layers + 1) * 64 + 4 * (total_x + total_a);
    p.table_bytes = (p.resid_at + 4 * most(H) + 127) / 128 * 128;
    p.xs_floats = (std::max(H, qd) + 31) / 32 * 32;
    const int scratch = std::max(p.xs_floats + step_scratch_floats(D, G), F);   // the MLP activations take the place of both
    const int fixed = step_shared_bytes() + p.table_bytes + (4 * scratch + 127) / 128 * 128;
    int chunk = ST_KV_BLOCK * D * (kv8 ? 2 : 4);
    for (const StepCols &c : p.cols) chunk = std::max(chunk, c.rows_per_chunk * c.K * 2);
    sl->max_chunk_bytes = (chunk + 127) / 128 * 128;
    const int ring = (smem_optin - fixed) / 128 * 128;
    if (ring < sl->max_chunk_bytes) return "model shape does not fit the shared memory";
    p.ring_bytes = ring;
    sl->dyn_smem = static_cast<size_t>(fixed) + ring;
    p.prefetch_bytes = ST_PREFETCH_BYTES;
    p.spin_limit = 1000000000u;   // 1 s
    const size_t chunks = static_cast<size_t>(std::max(1, grid / nkv));
    sl->ll_bytes = 8 * (static_cast<size_t>(grid) * (2 * p.x_line + p.q_line + p.ao_line + 16) + (static_cast<size_t>(F) + 15) / 16 * 16 + chunks * qd + chunks * nq * 2);
    return nullptr;
}
// Wire the exchange buffers (256-byte aligned base).
inline void step_wire(StepLaunch *sl, unsigned long long *base) {
    StepParams &p = sl->p;
    const size_t g = static_cast<size_t>(sl->grid), chunks = static_cast<size_t>(std::max(1, sl->grid / p.nkv));
    p.x_ll = base; base += g * p.x_line;
    p.xo_ll = base; base += g * p.x_line;
    p.q_ll = base; base += g * p.q_line;
    p.ao_ll = base; base += g * p.ao_line;
    p.lm_ll = base; base += g * 16;
    p.act_ll = base; base += (static_cast<size_t>(p.F) + 15) / 16 * 16;
    p.part_ll = base; base += chunks * p.qd;
    p.stat_ll = base;
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
