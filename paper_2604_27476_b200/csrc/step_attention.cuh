// Attention of the decode-step kernel: this CTA's chunk of the cached positions, the merge of the chunks.
#pragma once
#include "step_products.cuh"

namespace edgefm {
namespace ST_NS {

// The group's heads are the rows of tensor-core products: scores[head][position] = Q K^T takes the 8 heads' first two bf16 pieces as rows
// 0-7 and 8-15 of one m16n8k16 and the third as the rows of another (24 bits of the query, as the fp32 query it was), and
// out[head][dim] = P V the same of the probabilities; K and V enter as they are cached (signed bytes are exact in bf16).  The scores'
// registers are P's operand as they stand.  (With packed FMAs the phase took 30 us per layer for 32768 positions of 4 x 7 heads of
// 128, 2.3 TB/s of K and V.)
//   A tile is 16 positions.  Which positions is free as long as K's rows, V's rows and P agree: a block of n positions falls into four
// quarters of R rows, and tile i takes rows 4 i .. 4 i + 3 of every quarter, so that the four lanes of a V operand read from four
// quarters; those lie 32 bytes further apart than their rows fill, and the reads are free of bank conflicts.
__device__ __forceinline__ uint32_t codes_bf16(uint32_t w, unsigned sel) {     // two signed bytes: (128 + low 7 bits) - (128 or 256)
    const uint32_t x = __byte_perm(w, 0x43434343u, sel), lo = x & 0xff7fff7fu, sign = x & 0xff80ff80u;
    uint32_t r;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(lo), "r"(sign));
    return r;
}
__device__ __forceinline__ uint32_t two_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// The split of a block of n cached positions (kv_block) in shared memory: K rows one behind the other, then the quarters of V.
struct KvBlock {
    int n, R, v_at, v_stride;
    __device__ __forceinline__ KvBlock(int n_, int row_bytes) : n(n_), R((n_ + 15) / 16 * 4), v_at((n_ * row_bytes + 127) / 128 * 128), v_stride(R * row_bytes + 32) {}
    __device__ __forceinline__ int bytes() const { return v_at + 4 * v_stride; }
};

template <int D, int G, bool Q8>
struct WarpAttention {
    static constexpr int KS = D / 16, ROW = Q8 ? D : 2 * D, WD = D / 64;    // a warp multiplies P by 64 dims of V: WD warps per tile
    uint32_t q[KS][3][2];             // pieces of the query of head lane / 4
    float o[8][4];                    // dims 16 (lane % 4) + 8 e + i of this lane's head: o[i][e] + o[i][e + 2]
    float m, l;                       // of this lane's head; l: of this lane's positions
    static __device__ __forceinline__ int dim_of(int k, int t) { return Q8 ? 64 * (k >> 2) + 16 * t + 4 * (k & 3) : 32 * (k >> 1) + 8 * t + 4 * (k & 1); }
    __device__ __forceinline__ void start(const unsigned char *qs, int lane) {
        const int g = lane >> 2, t = lane & 3;
#pragma unroll
        for (int k = 0; k < KS; ++k)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const uint2 w = g < G ? *reinterpret_cast<const uint2 *>(qs + ((i * G + g) * D + dim_of(k, t)) * 2) : make_uint2(0u, 0u);
                q[k][i][0] = w.x;
                q[k][i][1] = w.y;
            }
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
        m = -INFINITY;
        l = 0.f;
    }
    // Tile i of a block; ks / vs: scales of this lane's four positions (compressed cache); dg: which 64 dims of V.
    __device__ __forceinline__ void tile(const unsigned char *kb, const unsigned char *vb, const KvBlock &b, int i, const float (&ks)[4], const float (&vs)[4], int dg, int lane) {
        const int g = lane >> 2, t = lane & 3, own = t * b.R + 4 * i;       // this lane's positions: own .. own + 3
        const bool odd = (g & 1) != 0;
        // V first: its loads fly while the scores are made
        uint32_t v[4][Q8 ? 2 : 4];
        const int last = b.n - 1, lq = (last >= b.R) + (last >= 2 * b.R) + (last >= 3 * b.R);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = own + k < b.n;                                  // (past the end: any row, its probability is zero)
            const unsigned char *row = vb + (in ? t : lq) * b.v_stride + (in ? 4 * i + k : last - lq * b.R) * ROW;
            if constexpr (Q8) {
                const uint2 w = *reinterpret_cast<const uint2 *>(row + dg * 64 + g * 8);
                v[k][0] = w.x; v[k][1] = w.y;
            } else {
                const uint4 w = *reinterpret_cast<const uint4 *>(row + dg * 128 + g * 16);
                v[k][0] = w.x; v[k][1] = w.y; v[k][Q8 ? 0 : 2] = w.z; v[k][Q8 ? 1 : 3] = w.w;
            }
        }
        float s[4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const unsigned char *row = kb + min((g >> 1) * b.R + 4 * i + (g & 1) + 2 * j, last) * ROW + t * 16;
            float a[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f};
            auto step = [&](int k, uint32_t b0, uint32_t b1) {
                mma(a, q[k][0][0], q[k][1][0], q[k][0][1], q[k][1][1], b0, b1);
                mma(e, q[k][2][0], 0u, q[k][2][1], 0u, b0, b1);
            };
            auto codes = [&](int k, uint32_t w) { step(k, codes_bf16(w, 0x4140), codes_bf16(w, 0x4342)); };
            // rows 128 bytes (or a multiple) apart start on the same bank: odd ones read the second 64 bytes first
            if constexpr (Q8 && D == 64) {
                const uint4 w = *reinterpret_cast<const uint4 *>(row);
                codes(0, w.x); codes(1, w.y); codes(2, w.z); codes(3, w.w);
            } else {
#pragma unroll
                for (int k = 0; k < ROW / 128; ++k) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(row + k * 128 + (odd ? 64 : 0)), y = *reinterpret_cast<const uint4 *>(row + k * 128 + (odd ? 0 : 64));
                    const uint4 w = pick(odd, x, y), z = pick(odd, y, x);
                    if constexpr (Q8) {
                        codes(0, w.x); codes(1, w.y); codes(2, w.z); codes(3, w.w);
                        codes(KS - 4, z.x); codes(KS - 3, z.y); codes(KS - 2, z.z); codes(KS - 1, z.w);
                    } else {
                        step(4 * k, w.x, w.y); step(4 * k + 1, w.z, w.w);
                        step(4 * k + 2, z.x, z.y); step(4 * k + 3, z.z, z.w);
                    }
                }
            }
            s[2 * j] = a[0] + a[2] + e[0];
            s[2 * j + 1] = a[1] + a[3] + e[1];
        }
        float mx = -INFINITY;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if constexpr (Q8) s[k] *= ks[k];
            if (own + k >= b.n) s[k] = -INFINITY;
            mx = fmaxf(mx, s[k]);
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        // the reference maximum moves only when it has grown by more than 2^8 (the probabilities may then reach 2^8)
        if (__any_sync(0xffffffffu, mx > m + 8.f)) {
            const float mn = fmaxf(m, mx), f = m == -INFINITY ? 0.f : exp2_approx(m - mn);
            l *= f;
            m = mn;
#pragma unroll
            for (int k = 0; k < 8; ++k) { o[k][0] *= f; o[k][1] *= f; o[k][2] *= f; o[k][3] *= f; }
        }
        uint32_t p[3][2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float x = exp2_approx(s[2 * j] - m), y = exp2_approx(s[2 * j + 1] - m);
            l += x + y;
            if constexpr (Q8) { x *= vs[2 * j]; y *= vs[2 * j + 1]; }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                p[k][j] = two_bf16(x, y);
                x -= bf16lo(p[k][j]);
                y -= bf16hi(p[k][j]);
            }
        }
        auto out = [&](int k, uint32_t b0, uint32_t b1) {
            mma(o[k], p[0][0], p[1][0], p[0][1], p[1][1], b0, b1);
            mma(o[k], p[2][0], 0u, p[2][1], 0u, b0, b1);
        };
        if constexpr (Q8) {
#pragma unroll
            for (int w = 0; w < 2; ++w)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t x = __byte_perm(v[0][w], v[1][w], h ? 0x7362 : 0x5140), y = __byte_perm(v[2][w], v[3][w], h ? 0x7362 : 0x5140);
                    out(4 * w + 2 * h, codes_bf16(x, 0x4140), codes_bf16(y, 0x4140));
                    out(4 * w + 2 * h + 1, codes_bf16(x, 0x4342), codes_bf16(y, 0x4342));
                }
        } else {
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                constexpr int Z = Q8 ? 1 : 3;
                out(2 * w, __byte_perm(v[0][w & Z], v[1][w & Z], 0x5410), __byte_perm(v[2][w & Z], v[3][w & Z], 0x5410));
                out(2 * w + 1, __byte_perm(v[0][w & Z], v[1][w & Z], 0x7632), __byte_perm(v[2][w & Z], v[3][w & Z], 0x7632));
            }
        }
    }
    // (m, l, o) to shared memory: mm, ml [NW][8], mo [NW][G][64]
    __device__ __forceinline__ void leave(float *mm, float *ml, float *mo, int warp, int lane) {
        const int g = lane >> 2, t = lane & 3;
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if (g >= G) return;
        if (t == 0) { mm[warp * 8 + g] = m; ml[warp * 8 + g] = l; }
        float *d = mo + (warp * G + g) * 64 + 16 * t;
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int i = 0; i < 8; i += 4)
                *reinterpret_cast<float4 *>(d + 8 * e + i) = make_float4(o[i][e] + o[i][e + 2], o[i + 1][e] + o[i + 1][e + 2], o[i + 2][e] + o[i + 2][e + 2], o[i + 3][e] + o[i + 3][e + 2]);
    }
};

// Shared-memory scratch of the attention, in floats: the queries' pieces | new k rows, new v rows (as cached), their scales | warp maxima,
// denominators, outputs.  The fp32 new rows share the place of the warp outputs.
template <int D, int G, int MT> struct AttScratch {
    static constexpr int QS = 0, NEW = QS + (3 * G * D / 2 + 3) / 4 * 4, NSC = NEW + MT * D, MM = NSC + 16, ML = MM + ST_NW * 8, MO = ML + ST_NW * 8,
                         RAW = 2 * MT * D, FLOATS = MO + (ST_NW * G * 64 > RAW ? ST_NW * G * 64 : RAW);
};

// Token share.tok, kv head share.g, the chunk [t0, t1) of the old positions; the last chunk also attends to the rows of the call's tokens
// 0 .. tok, which travel as packets.
template <int D, int G, bool Q8, int MT>
__device__ __forceinline__ bool attend(Ctx<MT> &c, int layer, const KvShare &share, unsigned tag) {
    using A = AttScratch<D, G, MT>;
    using W = WarpAttention<D, G, Q8>;
    const StepParams &p = c.p();
    float *base = reinterpret_cast<float *>(c.area());
    constexpr int half = D / 2;
    const int n_units = (p.nq + 2 * p.nkv) * half, n_new = share.tail ? share.tok + 1 : 0;
    bool ok = true;
    // queries of the group, then the new k and v rows: one row pair per packet pair
    constexpr int q_units = G * half, U = 3;                  // in flight per thread
    const int mine = q_units + n_new * 2 * half;
#pragma unroll 1
    for (int jb = 0; jb < mine; jb += U * ST_NT) {
        const int j0 = jb + c.tid;
        Two t[U];
        const unsigned long long *at[U];
        unsigned todo = 0;
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int j = j0 + i * ST_NT, kv = j - q_units;
            at[i] = p.q_ll;
            if (j < mine) {
                const int row = kv < 0 ? share.g * G * half + j : (kv & half) ? (p.nq + p.nkv + share.g) * half + (kv & (half - 1)) : (p.nq + share.g) * half + (kv & (half - 1));
                const int tok = kv < 0 ? share.tok : kv / (2 * half);
                const int w = ((row + 1) * c.ncta - 1) / n_units;      // its writer: the CTA c with first(c) <= row < first(c + 1)
                at[i] = p.q_ll + (static_cast<size_t>(tok) * c.ncta + w) * p.q_line + 2 * (row - st_first(n_units, w, c.ncta));
                todo |= 1u << i;
            }
        }
        const unsigned all = todo;
        Spin sp;
        int more;
        do {
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) t[i] = get2(at[i]);
#pragma unroll
            for (int i = 0; i < U; ++i)
                if ((todo >> i & 1u) && both(t[i], tag)) todo &= ~(1u << i);
            more = warp_again(sp, todo != 0u, c.abort(), p.spin_limit);
        } while (more > 0);
        if (more == 0) { ok = false; break; }
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (all >> i & 1u) {
                const int j = j0 + i * ST_NT, kv = j - q_units;
                const float lo = packet_value(t[i].a), hi = packet_value(t[i].b);
                if (kv < 0) {
                    unsigned char *d = reinterpret_cast<unsigned char *>(base + A::QS) + ((j / half) * D + (j & (half - 1))) * 2;
                    float x = lo * p.q_scale, y = hi * p.q_scale;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const uint32_t w = two_bf16(x, y);
                        store_u16(d + k * G * D * 2, static_cast<uint16_t>(w));
                        store_u16(d + k * G * D * 2 + half * 2, static_cast<uint16_t>(w >> 16));
                        x -= bf16lo(w);
                        y -= bf16hi(w);
                    }
                } else {
                    const int at_row = ((kv & half) ? n_new : 0) + kv / (2 * half);       // k rows, then v rows
                    if constexpr (Q8) {          // fp32 for the compression below
                        float *d = base + A::MO + at_row * D + (kv & (half - 1));
                        d[0] = lo;
                        d[half] = hi;
                    } else {
                        uint16_t *d = reinterpret_cast<uint16_t *>(base + A::NEW) + at_row * D + (kv & (half - 1));
                        d[0] = f32_to_bf16_bits(lo);
                        d[half] = f32_to_bf16_bits(hi);
                    }
                }
            }
    }
    if (!cta_vote(ok)) return false;
    if constexpr (Q8) {
        if (n_new > 0) {                // compress the new rows, a warp per row; the last one (this token's own) also goes to the cache
#pragma unroll 1
            for (int r = c.warp; r < 2 * n_new; r += ST_NW) {
                constexpr int DV = D / 32;
                const float *src = base + A::MO + r * D + c.lane * DV;
                float xv[DV], amax = 0.f;
#pragma unroll
                for (int e = 0; e < DV; ++e) { xv[e] = src[e]; amax = fmaxf(amax, fabsf(xv[e])); }
                amax = warp_max(amax);
                const float inv = amax > 0.f ? __fdiv_rn(127.0f, amax) : 0.f;
                uint32_t packed = 0u;
#pragma unroll
                for (int e = 0; e < DV; ++e) {
                    const float q = fminf(fmaxf(rintf(__fmul_rn(xv[e], inv)), -127.f), 127.f);
                    packed |= (static_cast<uint32_t>(static_cast<int>(q)) & 0xffu) << (8 * e);
                }
                const float sc = amax > 0.f ? __fdiv_rn(amax, 127.0f) : 0.f;
                const bool is_v = r >= n_new;
                const int k = is_v ? r - n_new : r;
                unsigned char *own = reinterpret_cast<unsigned char *>(base + A::NEW) + r * D + c.lane * DV;
                const size_t row = (static_cast<size_t>(layer) * p.nkv + share.g) * p.max_context + c.sh().n_old + k;
                unsigned char *dst = reinterpret_cast<unsigned char *>(is_v ? p.v_cache : p.k_cache) + row * D + c.lane * DV;
                if constexpr (DV == 4) { *reinterpret_cast<uint32_t *>(own) = packed; if (k == share.tok) *reinterpret_cast<uint32_t *>(dst) = packed; }
                else { *reinterpret_cast<uint16_t *>(own) = static_cast<uint16_t>(packed); if (k == share.tok) *reinterpret_cast<uint16_t *>(dst) = static_cast<uint16_t>(packed); }
                if (c.lane == 0) { base[A::NSC + (is_v ? 8 : 0) + k] = sc; if (k == share.tok) (is_v ? p.v_scale : p.k_scale)[row] = sc; }
            }
            if (!cta_vote(true)) return false;
        }
    }
    W att;
    att.start(reinterpret_cast<const unsigned char *>(base + A::QS), c.lane);
    const int my_tile = c.warp / W::WD, dg = c.warp & (W::WD - 1), quad = c.lane & 3;
    // (the new rows come last, by the last warps of the CTA that ends with them)
#pragma unroll 1
    for (int t = share.t0;; t += kv_positions(p, D)) {
        const bool fresh = t >= share.t1;
        if (fresh && n_new == 0) break;
        KvBlock b(fresh ? n_new : min(kv_positions(p, D), share.t1 - t), W::ROW);
        const int i = fresh ? ST_NW / W::WD - 1 - my_tile : my_tile, own = quad * b.R + 4 * i;
        const bool on = 4 * i < b.R;
        float ks[4] = {0.f, 0.f, 0.f, 0.f}, vs[4] = {0.f, 0.f, 0.f, 0.f};
        const unsigned char *at = reinterpret_cast<const unsigned char *>(base + A::NEW);
        if constexpr (Q8) {             // the scales of this lane's positions, asked for before the rows are awaited
            const size_t row = (static_cast<size_t>(layer) * p.nkv + share.g) * p.max_context + t + own;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (on && own + k < b.n) {
                    ks[k] = fresh ? base[A::NSC + own + k] : __ldcg(p.k_scale + row + k);
                    vs[k] = fresh ? base[A::NSC + 8 + own + k] : __ldcg(p.v_scale + row + k);
                }
        }
        if (fresh) {
            b.v_at = n_new * W::ROW;
            b.v_stride = b.R * W::ROW;
        } else if (!chunk_wait(c, at)) {
            ok = false;
            break;
        }
        if (on) att.tile(at, at + b.v_at, b, i, ks, vs, dg, c.lane);
        if (fresh) break;
        chunk_release(c);
    }
    att.leave(base + A::MM, base + A::ML, base + A::MO, c.warp, c.lane);
    if (!cta_vote(ok)) return false;
    // merge the warps and publish: one pair of dims per thread
    const size_t slot = static_cast<size_t>(share.tok) * c.sh().n_chunks + share.chunk;
#pragma unroll 1
    for (int j = c.tid; j < G * half; j += ST_NT) {
        const int h = j / half, d2 = j - h * half, dg = D == 64 ? 0 : d2 >> 5;      // (dims of group dg: every WD-th warp)
        float mw[ST_NW / W::WD], mm = -INFINITY;
#pragma unroll
        for (int w = 0; w < ST_NW / W::WD; ++w) { mw[w] = base[A::MM + w * W::WD * 8 + h]; mm = fmaxf(mm, mw[w]); }
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int w = 0; w < ST_NW / W::WD; ++w) {
            const float e = exp2_approx(mw[w] - mm);
            const float2 v = *reinterpret_cast<const float2 *>(base + A::MO + ((w * W::WD + dg) * G + h) * 64 + 2 * (d2 & 31));
            a = fmaf(v.x, e, a);
            b = fmaf(v.y, e, b);
        }
        put2(p.part_ll + slot * p.qd + (share.g * G + h) * D + 2 * d2, a, b, tag);
    }
    if (c.tid < G) {                    // maximum and denominator of every head, one store
        float mm = -INFINITY, ll = 0.f;
#pragma unroll
        for (int w = 0; w < ST_NW; w += W::WD) mm = fmaxf(mm, base[A::MM + w * 8 + c.tid]);
#pragma unroll
        for (int w = 0; w < ST_NW; w += W::WD) ll = fmaf(base[A::ML + w * 8 + c.tid], exp2_approx(base[A::MM + w * 8 + c.tid] - mm), ll);
        put2(p.stat_ll + (slot * p.nq + share.g * G + c.tid) * 2, mm, ll, tag);
    }
    return true;
}
// The owner of an output pair merges its chunks, in a fixed order: LP lanes per (token, pair), lanes over chunks.
template <int MT>
__device__ __forceinline__ bool merge_chunks(Ctx<MT> &c, unsigned tag) {
    constexpr int NJ = 3;                // chunks per lane in flight
    const StepParams &p = c.p();
    const int n_chunks = c.sh().n_chunks, m = c.sh().m;
    const int pairs = p.qd / 2, a0 = st_first(pairs, c.cta, c.ncta), n_pairs = st_first(pairs, c.cta + 1, c.ncta) - a0;
    // (several tokens: as few lanes as hold the chunks, so that all outputs are merged in one round)
    const int lp = MT == 1 || n_chunks > 16 * NJ ? 32 : n_chunks > 8 * NJ ? 16 : 8, sub = c.lane & (lp - 1), per_warp = 32 / lp;
    bool ok = true;
#pragma unroll 1
    for (int it = c.warp * per_warp; it < n_pairs * m && ok; it += ST_NW * per_warp) {
        const int item = it + c.lane / lp;
        const bool on = item < n_pairs * m;
        const int tok = on ? item / n_pairs : 0, k_pair = on ? item - tok * n_pairs : 0, pr = a0 + k_pair, h = 2 * pr / p.D;
        float mx = -INFINITY, l = 0.f, a = 0.f, b = 0.f;      // of this lane's chunks
#pragma unroll 1
        for (int kb = 0; kb < n_chunks; kb += lp * NJ) {
            const int k0 = kb + sub;
            Two st[NJ], ov[NJ];
            unsigned todo = 0;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                if (on && k0 + lp * j < n_chunks) todo |= 1u << j;
            const unsigned mine = todo;
            Spin sp;
            int more;
            do {
#pragma unroll
                for (int j = 0; j < NJ; ++j)
                    if (todo >> j & 1u) {
                        const size_t k = static_cast<size_t>(tok) * n_chunks + k0 + lp * j;
                        st[j] = get2(p.stat_ll + (k * p.nq + h) * 2);
                        ov[j] = get2(p.part_ll + k * p.qd + 2 * pr);
                    }
#pragma unroll
                for (int j = 0; j < NJ; ++j)
                    if ((todo >> j & 1u) && both(st[j], tag) && both(ov[j], tag)) todo &= ~(1u << j);
                more = warp_again(sp, todo != 0u, c.abort(), p.spin_limit);
            } while (more > 0);
            if (more == 0) { ok = false; break; }
            float mn = mx;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                if (mine >> j & 1u) mn = fmaxf(mn, packet_value(st[j].a));
            const float f = mx == -INFINITY ? 0.f : exp2_approx(mx - mn);      // (a lane without chunks keeps -inf)
            l *= f; a *= f; b *= f;
            mx = mn;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                if (mine >> j & 1u) {
                    const float e = exp2_approx(packet_value(st[j].a) - mn);
                    l = fmaf(packet_value(st[j].b), e, l);
                    a = fmaf(packet_value(ov[j].a), e, a);
                    b = fmaf(packet_value(ov[j].b), e, b);
                }
        }
        float mm = mx;
        for (int k = lp >> 1; k; k >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, k));
        const float f = mx == -INFINITY ? 0.f : exp2_approx(mx - mm);
        l *= f; a *= f; b *= f;
        for (int k = lp >> 1; k; k >>= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, k);
            a += __shfl_xor_sync(0xffffffffu, a, k);
            b += __shfl_xor_sync(0xffffffffu, b, k);
        }
        if (on && sub == 0) *reinterpret_cast<float2 *>(c.merged(tok) + 2 * k_pair) = make_float2(a / l, b / l);
    }
    if (!cta_vote(ok)) return false;
    if constexpr (st_packets(MT)) {
        // a line is written by one instruction: every further write invalidates the pollers' copies of it (+ 1.5 us)
        const unsigned real_tag = tag ^ c.sh().odd;
#pragma unroll 1
        for (int i = c.tid; i < n_pairs * MT; i += ST_NT) {        // (unused tokens too: their slots keep up with the tags)
            const int tok = i / n_pairs, k = i - tok * n_pairs;
            const float2 v = tok < m ? *reinterpret_cast<const float2 *>(c.merged(tok) + 2 * k) : make_float2(0.f, 0.f);
            put_raw2(p.ao_ll + (static_cast<size_t>(tok) * c.ncta + c.cta) * p.ao_line + 2 * k, pieces_packet(v.x, real_tag), pieces_packet(v.y, real_tag));
        }
    } else {
        const int stride = st_array_bytes(p.qd);
#pragma unroll 1
        for (int i = c.tid; i < 2 * n_pairs * m; i += ST_NT) {
            const int tok = i / (2 * n_pairs), k = i - tok * 2 * n_pairs;
            store_pieces<MT>(p.ao_vec, tok, 2 * a0 + k, stride, c.merged(tok)[k]);
        }
    }
    return true;
}

}  // namespace ST_NS
}  // namespace edgefm
