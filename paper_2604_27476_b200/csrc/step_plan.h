// Host-side tile schedules (edgefm_debug_plan_operator) and the tensor-map encoder of the prompt path.
//
// A schedule deals the rows of a matrix-vector operator out to CTAs and consumer warps as tiles of up to 16 rows x 256 columns.
// Every weight matrix is row-major bf16 [rows][K].  A CTA owns a contiguous range of the "units" of every operator (a
// unit is an output row; for the QKV and gate/up operators a pair of rows whose sums meet in one epilogue: the rotate-half
// RoPE partners i, i + d/2 of a head, or gate row i and up row F + i).  The range is cut into blocks of up to 16 rows (8
// pairs), every block into tiles of 256 columns, and the tiles, in (block, column) order, into one contiguous run per
// consumer warp.  Runs that cover all columns of a block finish the rows in the warp, the others leave partial sums in slots that
// are added in slot order (deterministic).
#pragma once
#include <cuda.h>   // CUtensorMap and its enums only: the encoder is looked up at run time, nothing links against the driver library
#include <cuda_runtime.h>
#include <stdint.h>
#include <algorithm>
#include <vector>

namespace edgefm {

constexpr int MK_PARTIAL_SLOTS = 48;   // partial sums a CTA has room for
constexpr int MK_TILE_COLS = 256, MK_TILE_ROWS = 16;
constexpr int MK_MAX_VARIANTS = 4;     // tile heights per matrix
enum { PH_QKV = 0, PH_RESID = 1, PH_SWIGLU = 2, PH_LMHEAD = 3 };

// 8 bytes per tile:
//   x: unit_base [0,20) | column piece [20,28) | height variant [28,30) | FIRST 30 | FLUSH 31
//   y: m [0,5) | first valid unit v0 [5,9) | DIRECT 9 | partial slot [10,20) | operator in layer (4 = output layer) [20,23) |
//      RAGGED 23 (K is not a multiple of 64)
// FIRST: a run of tiles starts.  FLUSH: it ends; DIRECT: the warp has seen all columns of these rows, otherwise the sums go to
// partial slot `slot`.
constexpr uint32_t MKT_FIRST = 1u << 30, MKT_FLUSH = 1u << 31, MKT_DIRECT = 1u << 9, MKT_RAGGED = 1u << 23;
inline uint2 mk_tile_desc(uint32_t unit_base, uint32_t kcol, uint32_t variant, bool first, bool flush, uint32_t m, uint32_t v0, bool direct,
                          uint32_t slot, uint32_t op, bool ragged) {
    uint2 d;
    d.x = (unit_base & 0xfffffu) | (kcol & 0xffu) << 20 | (variant & 3u) << 28 | (first ? MKT_FIRST : 0u) | (flush ? MKT_FLUSH : 0u);
    d.y = (m & 31u) | (v0 & 15u) << 5 | (direct ? MKT_DIRECT : 0u) | (slot & 1023u) << 10 | (op & 7u) << 20 | (ragged ? MKT_RAGGED : 0u);
    return d;
}
// Units whose row sums were left in partial slots: unit_base, m | v0 << 8, first slot, number of slots.
using MkCombine = uint4;

struct OpShape {
    int kind = 0;        // PH_*
    int units = 0;       // rows, or row pairs
    int K = 0;           // columns
    int rows = 0;        // rows of the matrix (tensor-map extent)
    int head_half = 0;   // PH_QKV: d / 2 (a block may not cross a head)
};

struct OpSchedule {
    int n_variants = 0;
    int variant_rows[MK_MAX_VARIANTS] = {0, 0, 0, 0};            // box heights of the operator's tensor maps
    std::vector<std::vector<std::vector<uint2>>> tiles;          // [cta][warp] tile list
    std::vector<std::vector<MkCombine>> combines;                // [cta]
    int max_slots = 0;                                           // partial slots the busiest CTA uses
};

inline bool op_paired(int kind) { return kind == PH_QKV || kind == PH_SWIGLU; }

// Schedule of one operator for `ncta` CTAs of `nw` consumer warps; slot_rows = rows a ring slot holds.
// op_index: 0..3 inside a layer, 4 = output layer.  Returns null, or why the operator does not fit.
inline const char *plan_op(const OpShape &os, int op_index, int ncta, int nw, int slot_rows, OpSchedule *out) {
    const bool paired = op_paired(os.kind);
    int B = paired ? std::min(8, slot_rows / 2) : std::min(MK_TILE_ROWS, slot_rows);   // units per block
    if (B < 1) return "ring slots too small for a tile";
    const int nkb = (os.K + MK_TILE_COLS - 1) / MK_TILE_COLS;
    if (nkb > 255) return "rows too long for the tile schedule";
    if (os.units >= (1 << 20)) return "too many rows for the tile schedule";
    OpSchedule &S = *out;
    S = OpSchedule();
    S.tiles.assign(ncta, std::vector<std::vector<uint2>>(nw));
    S.combines.assign(ncta, {});
    auto variant_of = [&](int rows, bool may_add) -> int {
        for (int v = 0; v < S.n_variants; ++v) if (S.variant_rows[v] == rows) return v;
        if (!may_add || S.n_variants == MK_MAX_VARIANTS) return -1;
        S.variant_rows[S.n_variants] = rows;
        return S.n_variants++;
    };
    // unit ranges of the CTAs.  QKV: in granules that divide a head's pairs, the granule that gives the smallest
    // largest share (so that blocks never cross a head and at most four box heights occur).
    int granule = 1;
    if (os.kind == PH_QKV) {
        long long best = -1;
        for (int g : {8, 4, 2}) {
            if (g > B || os.head_half % g) continue;
            const long long ng = os.units / g;
            const long long worst = ((ng + ncta - 1) / ncta) * g;
            if (best < 0 || worst < best) { best = worst; granule = g; }
        }
        if (best < 0) granule = 1;
        if (os.units % granule) return "QKV rows do not split into blocks";
        B = B / granule * granule;   // blocks of whole granules: at most four different heights (granule, 2 granules, ...)
    }
    struct Block { int u0, m, v0, variant; };
    for (int c = 0; c < ncta; ++c) {
        const long long ng = os.units / granule;
        const int u0 = static_cast<int>(ng * c / ncta) * granule, u1 = static_cast<int>(ng * (c + 1) / ncta) * granule;
        std::vector<Block> blocks;
        int u = u0;
        while (u < u1) {
            int m = std::min(B, u1 - u);
            if (os.kind == PH_QKV) m = std::min(m, os.head_half - u % os.head_half);   // stay inside the head
            int v = variant_of(m, true), v0 = 0, ub = u;
            if (v < 0) {
                // no tensor map of this height left: take a full block that ends where this one ends; its first units
                // repeat units that are already covered and are skipped in the epilogue
                if (os.kind == PH_QKV || u + m - B < u0) return "too many tile heights for one operator";
                v = variant_of(B, false);
                if (v < 0) return "too many tile heights for one operator";
                ub = u + m - B; v0 = B - m; m = B;
            }
            blocks.push_back({ub, m, v0, v});
            u = ub + m;
        }
        // tiles in (block, column) order, one contiguous run per warp
        const int T = static_cast<int>(blocks.size()) * nkb;
        int next_slot = 0;
        std::vector<int> first_slot(blocks.size(), -1), n_slots(blocks.size(), 0);
        for (int w = 0; w < nw; ++w) {
            const int t0 = static_cast<int>(static_cast<long long>(T) * w / nw), t1 = static_cast<int>(static_cast<long long>(T) * (w + 1) / nw);
            int t = t0;
            while (t < t1) {
                const int b = t / nkb, k0 = t % nkb;
                const int k1 = std::min(nkb, k0 + (t1 - t));        // columns [k0, k1) of block b
                const bool direct = k0 == 0 && k1 == nkb;
                int slot = 0;
                if (!direct) {
                    slot = next_slot++;
                    if (first_slot[b] < 0) first_slot[b] = slot;
                    ++n_slots[b];
                }
                for (int k = k0; k < k1; ++k)
                    S.tiles[c][w].push_back(mk_tile_desc(blocks[b].u0, k, blocks[b].variant, k == k0, k == k1 - 1, blocks[b].m, blocks[b].v0,
                                                         direct, slot, op_index, os.K % 64 != 0));
                t += k1 - k0;
            }
        }
        for (size_t b = 0; b < blocks.size(); ++b)
            if (n_slots[b] > 0)
                S.combines[c].push_back(make_uint4(static_cast<unsigned>(blocks[b].u0), static_cast<unsigned>(blocks[b].m | blocks[b].v0 << 8),
                                                   static_cast<unsigned>(first_slot[b]), static_cast<unsigned>(n_slots[b])));
        S.max_slots = std::max(S.max_slots, next_slot);
    }
    if (S.max_slots > MK_PARTIAL_SLOTS) return "too many partial sums per CTA";
    return nullptr;
}

// ---- tensor maps ---------------------------------------------------------------------------------------------------
using TensorMapEncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                       const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline TensorMapEncodeFn tensor_map_encoder() {
    static TensorMapEncodeFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<TensorMapEncodeFn>(p);
    }();
    return fn;
}

}  // namespace edgefm
