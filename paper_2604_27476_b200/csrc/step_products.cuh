// Staging of the input vectors and the matrix-vector products of the decode-step kernel.
#pragma once
#include "step_prims.cuh"

namespace edgefm {
namespace step {

// Place of value j of a staged vector of 8 * k8 values: two planes of 16-byte halves of its pieces, so that neighbouring lanes read
// neighbouring 16 bytes.
__device__ __forceinline__ int xs_at(int j, int k8) { return ((j & 4) ? k8 * 4 : 0) + (j >> 3) * 4 + (j & 3); }

// ---- exchanges: everybody reads a vector that lies in lines ---------------------------------------------------------------
// Table of the 16-byte units of such a vector: row | values << 16 | unit << 18 (unit = index of the packet pair).
// The tables of the residual stream and of the attention output stand in shared memory, made once per launch.
__device__ __forceinline__ int line_units(int n, int ncta, int grain) { return ((n / grain + ncta - 1) / ncta * grain + 1) / 2; }
__device__ __forceinline__ void make_table(const Ctx &c, unsigned *tab, int n, int grain, int line) {
    const int upl = line_units(n, c.ncta, grain), total = c.ncta * upl;
#pragma unroll 1
    for (int i = c.tid; i < total; i += ST_NT) {
        const int w = i / upl, e = i - w * upl;
        const int r0 = st_first(n / grain, w, c.ncta) * grain, r1 = st_first(n / grain, w + 1, c.ncta) * grain, row = r0 + 2 * e;
        tab[i] = static_cast<unsigned>(row & 0xffff) | static_cast<unsigned>(max(0, min(2, r1 - row))) << 16 | static_cast<unsigned>(w * (line >> 1) + e) << 18;
    }
}
__device__ __forceinline__ bool staged(Ctx &c, bool ok, float ss) {      // publish the sums of squares, meet
    ss = warp_sum(ss);
    if (c.lane == 0) c.sh().ss[c.warp] = ss;
    return cta_vote(ok);
}
// First operator of the step: the embedding row is the residual stream.
__device__ __forceinline__ bool stage_embedding(Ctx &c, const uint16_t *norm_w) {
    const StepParams &p = c.p();
    const uint16_t *erow = p.embed + static_cast<size_t>(c.sh().token) * p.H;
    float ss = 0.f;
#pragma unroll 1
    for (int i = c.tid; i < p.H; i += ST_NT) {
        const float v = bf16_bits_to_f32(erow[i]);
        ss = fmaf(v, v, ss);
        c.xs()[xs_at(i, p.H / 8)] = v * bf16_bits_to_f32(norm_w[i]);
    }
    return staged(c, true, ss);
}
// Wait for all values of the vector, times norm_w (RMSNorm weight, or null), into xs, and meet.
__device__ __forceinline__ bool stage_lines(Ctx &c, const unsigned *tab, int total, int k8, const unsigned long long *ll, const uint16_t *norm_w,
                                            unsigned tag) {
    constexpr int U = 4;     // units in flight per thread
    float *xs = c.xs();
    float ss = 0.f;
    bool ok = true;
#pragma unroll 1
    for (int base = c.tid; base < total; base += U * ST_NT) {
        unsigned e[U];
        float w0[U], w1[U];
        Two t[U];
        unsigned todo = 0;
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int u = base + i * ST_NT;
            e[i] = u < total ? tab[u] : 0u;
            const int cnt = (e[i] >> 16) & 3u;
            w0[i] = w1[i] = 1.f;
            if (cnt) {
                todo |= 1u << i;
                if (norm_w) {
                    w0[i] = bf16_bits_to_f32(__ldg(norm_w + (e[i] & 0xffffu)));
                    if (cnt > 1) w1[i] = bf16_bits_to_f32(__ldg(norm_w + (e[i] & 0xffffu) + 1));
                }
            }
        }
        Spin sp;
        for (;;) {
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) t[i] = get2(ll + static_cast<size_t>(e[i] >> 18) * 2);
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) {
                    const bool two = (e[i] >> 16 & 3u) > 1;
                    if (packet_tag(t[i].a) == tag && (!two || packet_tag(t[i].b) == tag)) {
                        todo &= ~(1u << i);
                        const int row = e[i] & 0xffffu;
                        const float a = packet_value(t[i].a);
                        ss = fmaf(a, a, ss);
                        xs[xs_at(row, k8)] = a * w0[i];
                        if (two) {
                            const float b = packet_value(t[i].b);
                            ss = fmaf(b, b, ss);
                            xs[xs_at(row + 1, k8)] = b * w1[i];
                        }
                    }
                }
            if (!todo) break;
            if (!sp.again(c.abort(), c.p().spin_limit)) { ok = false; break; }
        }
        if (!ok) break;
    }
    return staged(c, ok, ss);
}
// The MLP activations: every warp waits for its own slice (as the products deal out the columns) and leaves it in xs.
__device__ __forceinline__ bool stage_slice(Ctx &c, const unsigned long long *ll, unsigned tag) {
    constexpr int U = 6;     // packet pairs in flight per lane
    const int k8 = c.p().cols[ST_DN].K8;
    const int v0 = (k8 * c.warp / ST_NW) * 4, v1 = (k8 * (c.warp + 1) / ST_NW) * 4;      // pairs of values
    bool ok = true;
#pragma unroll 1
    for (int base = v0 + c.lane; base < v1; base += U * 32) {
        Two t[U];
        unsigned todo = 0;
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (base + i * 32 < v1) todo |= 1u << i;
        Spin sp;
        for (;;) {
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) t[i] = get2(ll + static_cast<size_t>(base + i * 32) * 2);
#pragma unroll
            for (int i = 0; i < U; ++i)
                if ((todo >> i & 1u) && both(t[i], tag)) {
                    todo &= ~(1u << i);
                    *reinterpret_cast<float2 *>(c.xs() + xs_at((base + i * 32) * 2, k8)) = make_float2(packet_value(t[i].a), packet_value(t[i].b));
                }
            if (!todo) break;
            if (!sp.again(c.abort(), c.p().spin_limit)) { ok = false; break; }
        }
        if (!ok) break;
    }
    return __all_sync(0xffffffffu, ok);
}

// ---- products ------------------------------------------------------------------------------------------------------------
// Rows [u, u1) (units) of operator `op`: this warp's column slice of every row, its sums to part[row][warp]; the input vector
// stands in xs.  PG pieces per lane are multiplied at once with ST row groups; up to PG pieces stay in registers for the whole
// operator, more are re-read for every group of rows.
struct Slice { int u, u1, op, batch; };

template <int PG, int ST>
__device__ __forceinline__ bool multiply(Ctx &c, const Slice &sl) {
    const StepParams &p = c.p();
    const StepCols &cols = p.cols[sl.op];
    float *const part = c.sh().part[sl.batch & 1];
    const int lpr_log2 = cols.lpr_log2, lpr = 1 << lpr_log2, rp = 32 >> lpr_log2;   // lanes of a row, rows at a time
    const int sub = c.lane & (lpr - 1), grp = c.lane >> lpr_log2;
    const int c0 = cols.K8 * c.warp / ST_NW + sub, c1 = cols.K8 * (c.warp + 1) / ST_NW, pieces = cols.pieces, k8 = cols.K8;
    const bool paired = op_paired(sl.op);
    const int row_bytes = cols.K * 2;
    const bool kept = pieces <= PG;
    const float *const xs = c.xs();
    f2 x[PG][4];
#pragma unroll
    for (int i = 0; i < PG; ++i) x[i][0] = x[i][1] = x[i][2] = x[i][3] = 0ull;      // (see Two)
    auto load_x = [&](int i0) {
#pragma unroll
        for (int i = 0; i < PG; ++i) {
            const int pc = c0 + ((i0 + i) << lpr_log2);
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (pc < c1) {
                a = *reinterpret_cast<const float4 *>(xs + pc * 4);
                b = *reinterpret_cast<const float4 *>(xs + (k8 + pc) * 4);
            }
            x[i][0] = pack2(a.x, a.y); x[i][1] = pack2(a.z, a.w); x[i][2] = pack2(b.x, b.y); x[i][3] = pack2(b.z, b.w);
        }
    };
    bool loaded = false;
    int done = 0;                              // units of this call finished
#pragma unroll 1
    for (int u = sl.u; u < sl.u1;) {
        const int n = chunk_units(p, sl.op, u, sl.u1), rows = paired ? 2 * n : n;
        const unsigned char *at;
        if (!chunk_wait(c, at)) return false;
#pragma unroll 1
        for (int s0 = 0; s0 < rows; s0 += rp * ST) {
            f2 acc[ST][2];
            const unsigned char *row[ST];
#pragma unroll
            for (int s = 0; s < ST; ++s) {
                row[s] = at + min(s0 + s * rp + grp, rows - 1) * row_bytes;
                acc[s][0] = acc[s][1] = 0ull;
            }
#pragma unroll 1
            for (int i0 = 0; i0 < pieces; i0 += PG) {
                if (!(kept && loaded)) load_x(i0);
                loaded = true;
                uint4 w[PG][ST];
#pragma unroll
                for (int i = 0; i < PG; ++i) {
                    const int off = min(c0 + ((i0 + i) << lpr_log2), k8 - 1) * 16;     // (past the slice: the vector is zero there)
#pragma unroll
                    for (int s = 0; s < ST; ++s) w[i][s] = *reinterpret_cast<const uint4 *>(row[s] + off);
                }
#pragma unroll
                for (int i = 0; i < PG; ++i)
#pragma unroll
                    for (int s = 0; s < ST; ++s) {
                        acc[s][0] = fma2(bf16x2_f2(w[i][s].x), x[i][0], acc[s][0]);
                        acc[s][1] = fma2(bf16x2_f2(w[i][s].y), x[i][1], acc[s][1]);
                        acc[s][0] = fma2(bf16x2_f2(w[i][s].z), x[i][2], acc[s][0]);
                        acc[s][1] = fma2(bf16x2_f2(w[i][s].w), x[i][3], acc[s][1]);
                    }
            }
            float sum[ST];
#pragma unroll
            for (int s = 0; s < ST; ++s) {
                const float2 a = unpack2(acc[s][0]), b = unpack2(acc[s][1]);
                sum[s] = (a.x + a.y) + (b.x + b.y);
            }
            const float v = fold<ST>(sum, sub, lpr);
            const int r = s0 + folded<ST>(sub, lpr) * rp + grp;
            if ((sub & (lpr / ST - 1)) == 0 && r < rows) part[(done + (r < n ? r : r - n + ST_BATCH)) * ST_NW + c.warp] = v;
        }
        chunk_release(c);
        u += n;
        done += n;
    }
    return true;
}
__device__ __forceinline__ bool multiply_any(Ctx &c, const Slice &sl) {
    switch (c.p().cols[sl.op].variant) {
        case ST_V14: return multiply<1, 4>(c, sl);
        case ST_V24: return multiply<2, 4>(c, sl);
        case ST_V34: return multiply<3, 4>(c, sl);
        case ST_V62: return multiply<6, 2>(c, sl);
        case ST_V101: return multiply<10, 1>(c, sl);
        default: return multiply<5, 2>(c, sl);
    }
}

}  // namespace step
}  // namespace edgefm
