// Staging of the input vectors and the matrix-vector products of the decode-step kernel.
#pragma once
#include "step_prims.cuh"

namespace edgefm {
namespace ST_NS {

// First operator of the step: the embedding rows are the residual streams; this CTA keeps its rows [x0, x0 + my_rows) of them.
// (The loads of U columns are under way together: one by one they took a trip to HBM each, 4 us for 1536 columns.)
template <int MT> __device__ __forceinline__ bool stage_embedding(Ctx<MT> &c, const uint16_t *norm_w, int x0, int my_rows) {
    constexpr int U = 8;
    const StepParams &p = c.p();
    const int stride = st_array_bytes(p.H), m = c.sh().m;
    zero_tail(c, p.H);
#pragma unroll 1
    for (int t = 0; t < m; ++t) {
        const uint16_t *erow = p.embed + static_cast<size_t>(c.sh().tokens[t]) * p.H;
        float ss = 0.f;
#pragma unroll 1
        for (int base = c.tid; base < p.H; base += U * ST_NT) {
            uint16_t e[U], w[U];
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int j = min(base + i * ST_NT, p.H - 1);
                e[i] = __ldg(erow + j);
                w[i] = __ldg(norm_w + j);
            }
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int j = base + i * ST_NT;
                if (j >= p.H) break;
                const float v = bf16_bits_to_f32(e[i]);
                ss = fmaf(v, v, ss);
                store_pieces<MT>(c.area(), t, j, stride, v * bf16_bits_to_f32(w[i]));
                if (j >= x0 && j < x0 + my_rows) c.resid()[t * my_rows + j - x0] = v;
            }
        }
        ss = warp_sum(ss);
        if (c.lane == 0) c.sh().merged[0][t * ST_NW + c.warp] = ss;      // (not in use yet)
    }
#pragma unroll 1
    for (int i = m * my_rows + c.tid; i < MT * my_rows; i += ST_NT) c.resid()[i] = 0.f;      // unused tokens
    if (!cta_vote(true)) return false;
    if (c.tid < m) c.sh().ss[c.tid] = sum8(&c.sh().merged[0][c.tid * ST_NW]);
    return true;
}
// Wait for a vector; sums: with the CTAs' sums of squares, which are added here (a warp per token).
template <int MT> __device__ __forceinline__ bool stage_vector(Ctx<MT> &c, bool sums) {
    if (!x_wait(c)) return false;
    if (sums && c.warp < c.sh().m) {
        const float *at = reinterpret_cast<const float *>(c.area() + Ctx<MT>::NA * st_array_bytes(c.p().H)) + c.warp * c.p().ss_stride;
        float ss = 0.f;
#pragma unroll 5
        for (int i = c.lane; i < c.ncta; i += 32) ss += at[i];
        ss = warp_sum(ss);
        if (c.lane == 0) c.sh().ss[c.warp] = ss;
    }
    x_release(c);
    return true;
}

// ---- exchanges: everybody reads a vector that lies in lines ---------------------------------------------------------------
// Table of the 16-byte units of such a vector: row | values | unit (unit = index of the packet pair).  The tables of the residual stream and of
// the attention output stand in shared memory, made once per launch (tight builds: in global memory, made by the host).
__device__ __forceinline__ int line_units(int n, int ncta, int grain) { return ((n / grain + ncta - 1) / ncta * grain + 1) / 2; }
// By `threads` threads, this one the `first`: a line each.
template <int MT> __device__ __forceinline__ void make_table(const Ctx<MT> &c, unsigned *tab, int n, int grain, int line, int first, int threads) {
    const int upl = line_units(n, c.ncta, grain);
#pragma unroll 1
    for (int w = first; w < c.ncta; w += threads) {
        int row = st_first(n / grain, w, c.ncta) * grain;
        const int r1 = st_first(n / grain, w + 1, c.ncta) * grain;
#pragma unroll 1
        for (int e = 0; e < upl; ++e, row += 2)
            tab[w * upl + e] = static_cast<unsigned>(row & ((1 << ROW_BITS) - 1)) | static_cast<unsigned>(max(0, min(2, r1 - row))) << ROW_BITS | static_cast<unsigned>(w * (line >> 1) + e) << (ROW_BITS + 2);
    }
}
// Wait for all values of the vectors of all tokens (K columns, lines of `line` packets) and leave their pieces in shared memory, and meet.
// sums: the last packet of every line is a partial sum of squares.
template <int MT>
__device__ __forceinline__ bool stage_lines(Ctx<MT> &c, const unsigned *tab, int total, int K, const unsigned long long *ll, int line, bool sums, unsigned tag) {
    constexpr int U = MT == 1 ? 4 : 7, W = 5;     // units in flight per thread; lines whose sums a lane reads together
    const int m = c.sh().m, all = m * total, stride = st_array_bytes(K);
    bool ok = true;
    // the sums of squares of token w are added by warp w; asked for first, awaited last
    const unsigned long long *const sums_at = ll + static_cast<size_t>(c.warp) * c.ncta * line + line - 1;
    const bool adds = sums && c.warp < m;
    unsigned long long s[W] = {0ull, 0ull, 0ull, 0ull, 0ull};
    auto ask = [&](int base) {
#pragma unroll
        for (int i = 0; i < W; ++i)
            if (base + 32 * i < c.ncta) s[i] = get1(sums_at + static_cast<size_t>(base + 32 * i) * line);
    };
    if (adds) ask(c.lane);
    zero_tail(c, K);
#pragma unroll 1
    for (int base0 = 0; base0 < all; base0 += U * ST_NT) {
        const int base = base0 + c.tid;
        unsigned e[U], at[U];
        Two t[U];
        unsigned todo = 0;
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int u = base + i * ST_NT;
            int tok = 0;
            if constexpr (MT > 1) tok = u / total;
            e[i] = u < all ? tab[u - tok * total] : 0u;
            at[i] = (e[i] >> (ROW_BITS + 2)) * 2 + static_cast<unsigned>(tok * c.ncta * line);
            e[i] = (e[i] & ((4u << ROW_BITS) - 1u)) | static_cast<unsigned>(tok) << (ROW_BITS + 2);
            if ((e[i] >> ROW_BITS) & 3u) todo |= 1u << i;
        }
        Spin sp;
        for (;;) {
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) t[i] = get2(ll + at[i]);
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) {
                    const bool two = (e[i] >> ROW_BITS & 3u) > 1;
                    if (pieces_tag(t[i].a, tag) && (!two || pieces_tag(t[i].b, tag))) {
                        todo &= ~(1u << i);
                        const int row = e[i] & ((1u << ROW_BITS) - 1u), tok = static_cast<int>(e[i] >> (ROW_BITS + 2));
                        store_packet<MT>(c.area(), tok, row, stride, t[i].a);
                        if (two) store_packet<MT>(c.area(), tok, row + 1, stride, t[i].b);
                    }
                }
            const int more = warp_again(sp, todo != 0u, c.abort(), c.p().spin_limit);
            if (more == 0) ok = false;
            if (more <= 0) break;
        }
        if (!ok) break;
    }
    if (adds) {
        float ss = 0.f;
#pragma unroll 1
        for (int base0 = 0; base0 < c.ncta && ok; base0 += 32 * W) {
            const int base = base0 + c.lane;
            if (base0 != 0) ask(base);
            Spin sp;
            for (;;) {
                bool here = true;
#pragma unroll
                for (int i = 0; i < W; ++i)
                    if (base + 32 * i < c.ncta) here = here && packet_tag(s[i]) == tag;
                const int more = warp_again(sp, !here, c.abort(), c.p().spin_limit);
                if (more == 0) ok = false;
                if (more <= 0) break;
                ask(base);
            }
#pragma unroll
            for (int i = 0; i < W; ++i)
                if (base + 32 * i < c.ncta) ss += packet_value(s[i]);
        }
        ss = warp_sum(ss);
        if (c.lane == 0) c.sh().ss[c.warp] = ss;
    }
    return cta_vote(ok);
}

// The MLP activations whole (K columns), from packets in natural order, four at a time (32-byte loads; K is a multiple of 8).  All of a
// round's loads are under way together: with pairs, 8960 columns took two rounds of polls.
template <int MT> __device__ __forceinline__ bool stage_activations(Ctx<MT> &c, unsigned tag) {
    constexpr int U = 9;     // quads in flight per thread
    const StepParams &p = c.p();
    const int K = p.F, quads = K / 4, all = c.sh().m * quads, stride = st_array_bytes(K);
    bool ok = true;
    zero_tail(c, K);
#pragma unroll 1
    for (int base0 = 0; base0 < all; base0 += U * ST_NT) {
        const int base = base0 + c.tid;
        Four t[U];
        unsigned todo = 0;
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (base + i * ST_NT < all) todo |= 1u << i;
        auto at = [&](int i) {
            const int u = base + i * ST_NT, tok = MT > 1 && u >= quads ? 1 : 0;
            return p.act_ll + static_cast<size_t>(tok) * p.act_len + 4 * (u - tok * quads);
        };
        Spin sp;
        for (;;) {
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) t[i] = get4(at(i));
#pragma unroll
            for (int i = 0; i < U; ++i)
                if ((todo >> i & 1u) && pieces_tag(t[i].a, tag) && pieces_tag(t[i].b, tag) && pieces_tag(t[i].c, tag) && pieces_tag(t[i].d, tag)) {
                    todo &= ~(1u << i);
                    const int u = base + i * ST_NT, tok = MT > 1 && u >= quads ? 1 : 0;
                    unsigned char *to = c.area() + tok * Ctx<MT>::S * stride + (u - tok * quads) * 8;
                    const uint32_t a0 = static_cast<uint32_t>(t[i].a), b0 = static_cast<uint32_t>(t[i].b), c0 = static_cast<uint32_t>(t[i].c), d0 = static_cast<uint32_t>(t[i].d);
                    const uint32_t a1 = static_cast<uint32_t>(t[i].a >> 32), b1 = static_cast<uint32_t>(t[i].b >> 32), c1 = static_cast<uint32_t>(t[i].c >> 32), d1 = static_cast<uint32_t>(t[i].d >> 32);
                    *reinterpret_cast<uint2 *>(to) = make_uint2(__byte_perm(a0, b0, 0x5410), __byte_perm(c0, d0, 0x5410));
                    *reinterpret_cast<uint2 *>(to + stride) = make_uint2(__byte_perm(a0, b0, 0x7632), __byte_perm(c0, d0, 0x7632));
                    *reinterpret_cast<uint2 *>(to + 2 * stride) = make_uint2(__byte_perm(a1, b1, 0x5410), __byte_perm(c1, d1, 0x5410));
                }
            const int more = warp_again(sp, todo != 0u, c.abort(), p.spin_limit);
            if (more == 0) ok = false;
            if (more <= 0) break;
        }
        if (!ok) break;
    }
    return cta_vote(ok);
}

// ---- products ------------------------------------------------------------------------------------------------------------
// One mma.m16n8k16 multiplies a 16-row x 16-column block of bf16 weights (A) by B = [16 x 8], whose columns are the pieces of the
// tokens' activations (token * S + piece); products of two bf16 values are exact in fp32, accumulation is fp32.  The instruction
// serves as a dot-product unit: 16 bytes of weights cost 8 conversions and 4 packed FMAs otherwise (measured from L2 over the
// chip, 48 KB chunks: 13 TB/s; this form 16 TB/s; the copies alone 19 TB/s; HBM 7 TB/s).
//   A lane reads 16 bytes (8 columns) of rows g = lane / 4 and g + 8 at piece t = lane % 4 of a 32-column half of a 64-column block:
// the four words are the A registers of two instructions (which columns a "k" stands for does not matter as long as B agrees:
// its lane (n = g, t) reads the same 16 bytes of array n).  All rows start on the same banks, so odd rows read the block's second
// half first and swap afterwards.
__device__ __forceinline__ void mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 pick(bool second, const uint4 &a, const uint4 &b) {
    return make_uint4(second ? b.x : a.x, second ? b.y : a.y, second ? b.z : a.z, second ? b.w : a.w);
}
template <int SETS> struct Acc {       // row sums of a tile: two independent chains per 8 B columns
    float d[SETS][2][4];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int s = 0; s < SETS; ++s)
#pragma unroll
            for (int q = 0; q < 2; ++q) d[s][q][0] = d[s][q][1] = d[s][q][2] = d[s][q][3] = 0.f;
    }
};
// A block (64 columns) of a chunk at offset `off`: rows ra / rb (this lane's), `last` = offset of the last 16 bytes of a row.
// HALF: there is no row rb (the lower half of the MMA is zero).
template <int SETS, bool HALF = false>
__device__ __forceinline__ void block_mma(Acc<SETS> &acc, const unsigned char *ra, const unsigned char *rb, int off, bool odd, int last, const uint4 (&b0)[SETS], const uint4 (&b1)[SETS]) {
    const int o0 = min(off + (odd ? 64 : 0), last), o1 = min(off + (odd ? 0 : 64), last);    // (past the row: the vector is zero there)
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const uint4 p0 = *reinterpret_cast<const uint4 *>(ra + o0), q0 = HALF ? zero : *reinterpret_cast<const uint4 *>(rb + o0);
    const uint4 p1 = *reinterpret_cast<const uint4 *>(ra + o1), q1 = HALF ? zero : *reinterpret_cast<const uint4 *>(rb + o1);
    const uint4 a = pick(odd, p0, p1), b = pick(odd, q0, q1), e = pick(odd, p1, p0), f = pick(odd, q1, q0);
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
        mma(acc.d[s][0], a.x, b.x, a.y, b.y, b0[s].x, b0[s].y);
        mma(acc.d[s][1], a.z, b.z, a.w, b.w, b0[s].z, b0[s].w);
        mma(acc.d[s][0], e.x, f.x, e.y, f.y, b1[s].x, b1[s].y);
        mma(acc.d[s][1], e.z, f.z, e.w, f.w, b1[s].z, b1[s].w);
    }
}
// The row sums of a finished tile to part[token][row][warp]; this lane's two MMA rows are rows ra and rb of the batch (-1: none).
template <int MT, int SETS>
__device__ __forceinline__ void flush(const Ctx<MT> &c, Acc<SETS> &acc, float *part, int ra, int rb) {
    const int t = c.lane & 3;
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
        float d[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = acc.d[s][0][e] + acc.d[s][1][e];
        if constexpr (Ctx<MT>::S == 2) {                  // columns 2 t, 2 t + 1 are the pieces of token 4 s + t
            float *at = part + (4 * s + t) * Ctx<MT>::RB * ST_NW + c.warp;
            if (4 * s + t < MT) {
                if (ra >= 0) at[ra * ST_NW] = d[0] + d[1];
                if (rb >= 0) at[rb * ST_NW] = d[2] + d[3];
            }
        } else {                                          // token 0: columns 0, 1, 2; token 1: columns 3, 4, 5
            const float n0 = __shfl_down_sync(0xffffffffu, d[0], 1), n2 = __shfl_down_sync(0xffffffffu, d[2], 1);
            float *at = part + c.warp;
            if (t == 0) {
                if (ra >= 0) at[ra * ST_NW] = d[0] + d[1] + n0;
                if (rb >= 0) at[rb * ST_NW] = d[2] + d[3] + n2;
            }
            if constexpr (MT == 2) {
                const float m0 = __shfl_down_sync(0xffffffffu, d[1], 1), m2 = __shfl_down_sync(0xffffffffu, d[3], 1);
                const float k0 = __shfl_down_sync(0xffffffffu, d[0] + d[1], 2), k2 = __shfl_down_sync(0xffffffffu, d[2] + d[3], 2);
                at += Ctx<MT>::RB * ST_NW;
                if (t == 0) {
                    if (ra >= 0) at[ra * ST_NW] = m0 + k0;
                    if (rb >= 0) at[rb * ST_NW] = m2 + k2;
                }
            }
        }
    }
}

// This lane's two rows of a chunk cut by columns: their first bytes, the distance of the 64-column blocks, the last readable offset.
struct Rows { const unsigned char *a, *b; int block, last; };
__device__ __forceinline__ Rows rows_of(const unsigned char *at, int g, int na, int nb, int row_bytes, bool paired, const StepCols &cols, int t16) {
    const int r0 = min(g, na - 1);
    if (cols.box_rows == 0) return Rows{at + r0 * row_bytes + t16, at + min(na + g, na + nb - 1) * row_bytes + t16, 128, row_bytes - 16 - t16};
    // boxes: [block][row][128 bytes]; the partners of a pair are a box of their own
    const int r1 = paired ? r0 : min(na + g, na + nb - 1);
    const unsigned char *second = paired ? at + cols.box_rows * cols.seg * 2 : at;
    return Rows{at + r0 * 128 + t16, second + r1 * 128 + t16, cols.box_rows * 128, 1 << 30};
}

struct Slice { int u, u1, op, batch; };      // units [u, u1) of an operator; the batch of partial sums they go to

// KEEP > 0: rows are whole in a chunk and a warp's blocks of the vector (at most KEEP) stay in registers for all tiles; more than
// ST_KEEP: tiles of 8 rows in all, the upper half of the MMA.
// KEEP == 0: tiles cut by columns, the vector is read again for every tile (the MLP activations come by segments themselves).
template <int KEEP, int MT>
__device__ __forceinline__ bool multiply(Ctx<MT> &c, const Slice &sl) {
    constexpr int SETS = (Ctx<MT>::NA + 7) / 8;
    constexpr bool HALF = KEEP > ST_KEEP;
    const StepParams &p = c.p();
    const int K = p.cols[sl.op].K, seg = p.cols[sl.op].seg;
    float *const part = c.sh().part[sl.batch & 1];
    const int g = c.lane >> 2, t16 = (c.lane & 3) * 16;
    const bool odd = (g & 1) != 0, paired = op_paired(sl.op), down = KEEP == 0 && sl.op == ST_DN && !p.act_packets;
    const int stride = st_array_bytes(down ? seg : K), slot = Ctx<MT>::NA * stride;
    const unsigned char *xb[SETS];           // this lane's array of the staged vector (columns of B past the last array: any)
#pragma unroll
    for (int s = 0; s < SETS; ++s) xb[s] = c.area() + min(8 * s + g, Ctx<MT>::NA - 1) * stride + t16;
    constexpr int NK = KEEP > 0 ? KEEP : 1;
    uint4 k0[NK][SETS], k1[NK][SETS];
    const int nb_all = (K + 63) / 64, first_all = nb_all * c.warp / ST_NW, mine_all = nb_all * (c.warp + 1) / ST_NW - first_all;
    if constexpr (KEEP > 0) {
#pragma unroll
        for (int i = 0; i < NK; ++i)
#pragma unroll
            for (int s = 0; s < SETS; ++s) {
                const bool on = i < mine_all;
                const unsigned char *at = xb[s] + (first_all + (on ? i : 0)) * 128;
                k0[i][s] = on ? *reinterpret_cast<const uint4 *>(at) : make_uint4(0u, 0u, 0u, 0u);
                k1[i][s] = on ? *reinterpret_cast<const uint4 *>(at + 64) : make_uint4(0u, 0u, 0u, 0u);
            }
    }
    Acc<SETS> acc;
    acc.clear();
#pragma unroll 1
    for (int u = sl.u; u < sl.u1;) {
        const int n = tile_units(p, sl.op, u, sl.u1);
        const int na = paired ? n : min(n, 8), nb = paired ? n : n - na;                       // rows in the upper and lower half of the MMA
        if constexpr (KEEP > 0) {
            const unsigned char *at;
            if (!chunk_wait(c, at)) return false;
            const int rb = K * 2;
            const unsigned char *ra = at + min(g, (HALF ? na + nb : na) - 1) * rb + t16 + first_all * 128, *rc = at + min(na + g, na + nb - 1) * rb + t16 + first_all * 128;
            const int last = rb - 16 - t16 - first_all * 128;
#pragma unroll
            for (int i = 0; i < NK; ++i)
                if (!HALF || i < mine_all) block_mma<SETS, HALF>(acc, ra, rc, i * 128, odd, last, k0[i], k1[i]);
            chunk_release(c);
        } else {
#pragma unroll 1
            for (int col = 0; col < K; col += seg) {
                const unsigned char *at;
                if (down && !x_wait(c)) return false;
                if (!chunk_wait(c, at)) return false;
                const int x_off = down ? c.act_slot * slot : col * 2;
                const int cols = min(seg, K - col), nblk = (cols + 63) / 64;
                const int j0 = nblk * c.warp / ST_NW, j1 = nblk * (c.warp + 1) / ST_NW;
                const Rows r = rows_of(at, g, na, nb, cols * 2, paired, p.cols[sl.op], t16);
#pragma unroll 2
                for (int j = j0; j < j1; ++j) {
                    uint4 b0[SETS], b1[SETS];
#pragma unroll
                    for (int s = 0; s < SETS; ++s) {
                        const unsigned char *x = xb[s] + x_off + j * 128;
                        b0[s] = *reinterpret_cast<const uint4 *>(x);
                        b1[s] = *reinterpret_cast<const uint4 *>(x + 64);
                    }
                    block_mma<SETS>(acc, r.a, r.b, j * r.block, odd, r.last, b0, b1);
                }
                chunk_release(c);
                if (down) {
                    x_release(c);
                    if (++c.act_slot == p.act_slots) c.act_slot = 0;
                }
            }
        }
        const int done = u - sl.u, second = paired ? Ctx<MT>::RB / 2 + done : done + 8;
        if constexpr (HALF) flush<MT, SETS>(c, acc, part, g < na ? done + g : g < na + nb ? second + g - na : -1, -1);
        else flush<MT, SETS>(c, acc, part, g < na ? done + g : -1, g < nb ? second + g : -1);
        acc.clear();
        u += n;
    }
    return true;
}

template <int MT> __device__ __forceinline__ bool multiply_any(Ctx<MT> &c, const Slice &sl) {
    const StepCols &cols = c.p().cols[sl.op];
    if (cols.segs > 1 || sl.op == ST_DN) return multiply<0, MT>(c, sl);
    const int most = ((cols.K + 63) / 64 + ST_NW - 1) / ST_NW;
    if constexpr (Ctx<MT>::NA <= 8)          // (with two sets of B columns the vector does not fit the registers)
        if (most > ST_KEEP && most <= ST_KEEP_HALF && cols.tile == (op_paired(sl.op) ? ST_TILE / 4 : ST_TILE / 2)) return multiply<ST_KEEP_HALF, MT>(c, sl);
    switch (most) {
        case 1: return multiply<1, MT>(c, sl);
        case 2: return multiply<2, MT>(c, sl);
        case 3: return multiply<3, MT>(c, sl);
        case 4: return multiply<4, MT>(c, sl);
        default: return multiply<0, MT>(c, sl);
    }
}

}  // namespace ST_NS
}  // namespace edgefm
