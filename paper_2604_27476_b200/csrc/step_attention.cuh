// Attention of the decode-step kernel: this CTA's chunk of the cached positions, the merge of the chunks.
#pragma once
#include "step_prims.cuh"

namespace edgefm {
namespace step {

// Queries of the group in registers (8 dims of every head per lane), K and V rows from the ring; every warp keeps a running
// reference maximum, denominator and output of its own positions.  A score is the dot product over the D / 8 lanes of a
// position, all heads folded at once, so that a lane ends up with the score of one (position, head).
__device__ __forceinline__ float code_f32(uint32_t u, unsigned sel) {     // byte + 128 in the mantissa of 2^23: a signed code, exactly
    return __uint_as_float(__byte_perm(u, 0x4B000000u, sel)) - 8388736.f;
}
__device__ __forceinline__ void codes8_to_f2(uint2 w, f2 (&f)[4]) {
    const uint32_t a = w.x ^ 0x80808080u, b = w.y ^ 0x80808080u;
    f[0] = pack2(code_f32(a, 0x7440), code_f32(a, 0x7441)); f[1] = pack2(code_f32(a, 0x7442), code_f32(a, 0x7443));
    f[2] = pack2(code_f32(b, 0x7440), code_f32(b, 0x7441)); f[3] = pack2(code_f32(b, 0x7442), code_f32(b, 0x7443));
}

template <int D, int G, bool Q8>
struct WarpAttention {
    static constexpr int LPR = D / 8, SP = 32 / LPR, DV = D / 32;   // eight positions per warp and block, SP at a time
    static constexpr int ROW = Q8 ? D : 2 * D;
    f2 q[G][4];
    f2 o[G][DV / 2];
    float m, l;                       // of this lane's head
    __device__ __forceinline__ void start(const float *qs, int lane) {
        const int sub = lane & (LPR - 1);
#pragma unroll
        for (int h = 0; h < G; ++h) {
            const float4 a = *reinterpret_cast<const float4 *>(qs + h * D + sub * 8), b = *reinterpret_cast<const float4 *>(qs + h * D + sub * 8 + 4);
            q[h][0] = pack2(a.x, a.y); q[h][1] = pack2(a.z, a.w); q[h][2] = pack2(b.x, b.y); q[h][3] = pack2(b.z, b.w);
#pragma unroll
            for (int e = 0; e < DV / 2; ++e) o[h][e] = 0ull;
        }
        m = -INFINITY;
        l = 0.f;
    }
    static __device__ __forceinline__ int head_of(int lane) { return folded<8>(lane & (LPR - 1), LPR); }
    // Positions [first, first + cnt) (cnt <= 8) of the block at kb / vb; ks / vs: scales of these rows (compressed cache);
    // pw: this warp's 8 x 8 probabilities.
    __device__ __forceinline__ void block(const unsigned char *kb, const unsigned char *vb, const float *ks, const float *vs, int first, int cnt, float *pw, int lane) {
        const int sub = lane & (LPR - 1), grp = lane / LPR, h_mine = head_of(lane);
        // (a loop, the scores parked in shared memory by the lane that needs them again: unrolled, the code of a layer outgrows the
        // instruction cache and every phase starts with misses)
        float mx = -INFINITY;
#pragma unroll 1
        for (int st = 0; st * SP < cnt; ++st) {
            const int pos = first + min(st * SP + grp, cnt - 1);
            f2 kf[4];
            if constexpr (Q8) {
                codes8_to_f2(*reinterpret_cast<const uint2 *>(kb + pos * ROW + sub * 8), kf);
            } else {
                const uint4 w = *reinterpret_cast<const uint4 *>(kb + pos * ROW + sub * 16);
                kf[0] = bf16x2_f2(w.x); kf[1] = bf16x2_f2(w.y); kf[2] = bf16x2_f2(w.z); kf[3] = bf16x2_f2(w.w);
            }
            float v[8];
#pragma unroll
            for (int h = 0; h < 8; ++h) {
                v[h] = 0.f;
                if (h < G) {
                    f2 a = fma2(kf[0], q[h < G ? h : 0][0], 0ull);
                    a = fma2(kf[1], q[h < G ? h : 0][1], a);
                    a = fma2(kf[2], q[h < G ? h : 0][2], a);
                    a = fma2(kf[3], q[h < G ? h : 0][3], a);
                    const float2 t = unpack2(a);
                    v[h] = t.x + t.y;
                }
            }
            float r = fold<8>(v, sub, LPR);
            if (Q8 && st * SP + grp < cnt) r *= ks[st * SP + grp];
            if (st * SP + grp >= cnt) r = -INFINITY;
            mx = fmaxf(mx, r);
            pw[(st * SP + grp) * 8 + h_mine] = r;
        }
#pragma unroll
        for (int k = LPR; k < 32; k <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, k));
        // the reference maximum moves only when it has grown by more than 2^8 (the probabilities may then reach 2^8)
        if (__any_sync(0xffffffffu, mx > m + 8.f)) {
            const float mn = fmaxf(m, mx), f = m == -INFINITY ? 0.f : exp2_approx(m - mn);
            l *= f;
            m = mn;
#pragma unroll
            for (int h = 0; h < G; ++h) {
                // a lane that holds head h: the bits of folded() from the top
                constexpr int S1 = LPR >> 1, S2 = LPR >> 2, S3 = LPR >> 3;
                const float fh = __shfl_sync(0xffffffffu, f, ((h & 4) ? S1 : 0) | ((h & 2) ? S2 : 0) | ((h & 1) ? S3 : 0));
                const f2 fh2 = pack2(fh, fh);
#pragma unroll
                for (int e = 0; e < DV / 2; ++e) o[h][e] = fma2(o[h][e], fh2, 0ull);
            }
        }
#pragma unroll 1
        for (int i = grp; i < cnt; i += SP) {
            const float pr = exp2_approx(pw[i * 8 + h_mine] - m);
            l += pr;
            pw[i * 8 + h_mine] = Q8 ? pr * vs[i] : pr;
        }
        __syncwarp();
#pragma unroll 2
        for (int i = 0; i < cnt; ++i) {
            f2 v[DV / 2];
            const unsigned char *row = vb + (first + i) * ROW;
            if constexpr (Q8) {
                uint32_t w;
                if constexpr (DV == 4) w = *reinterpret_cast<const uint32_t *>(row + lane * 4);
                else w = *reinterpret_cast<const uint16_t *>(row + lane * 2);
                const uint32_t u = w ^ 0x80808080u;
#pragma unroll
                for (int e = 0; e < DV / 2; ++e) v[e] = pack2(code_f32(u, 0x7440 + 2 * e), code_f32(u, 0x7441 + 2 * e));
            } else if constexpr (DV == 4) {
                const uint2 w = *reinterpret_cast<const uint2 *>(row + lane * 8);
                v[0] = bf16x2_f2(w.x);
                v[DV / 2 - 1] = bf16x2_f2(w.y);
            } else {
                v[0] = bf16x2_f2(*reinterpret_cast<const uint32_t *>(row + lane * 4));
            }
            const float4 pa = *reinterpret_cast<const float4 *>(pw + i * 8), pb = *reinterpret_cast<const float4 *>(pw + i * 8 + 4);
            const float pr[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const f2 pp = pack2(pr[h], pr[h]);
#pragma unroll
                for (int e = 0; e < DV / 2; ++e) o[h][e] = fma2(pp, v[e], o[h][e]);
            }
        }
        __syncwarp();
    }
    // (m, l, o) to shared memory: mm, ml [NW][8], mo [NW][G][D]
    __device__ __forceinline__ void leave(float *mm, float *ml, float *mo, int warp, int lane) {
        float lt = l;
#pragma unroll
        for (int k = LPR; k < 32; k <<= 1) lt += __shfl_xor_sync(0xffffffffu, lt, k);
        if (lane < LPR) { mm[warp * 8 + head_of(lane)] = m; ml[warp * 8 + head_of(lane)] = lt; }
#pragma unroll
        for (int h = 0; h < G; ++h) {
            float *d = mo + (warp * G + h) * D + lane * DV;
            if constexpr (DV == 4) {
                const float2 a = unpack2(o[h][0]), b = unpack2(o[h][DV / 2 - 1]);
                *reinterpret_cast<float4 *>(d) = make_float4(a.x, a.y, b.x, b.y);
            } else {
                *reinterpret_cast<float2 *>(d) = unpack2(o[h][0]);
            }
        }
    }
};

// Shared-memory scratch of the attention, in floats: queries | new k rows, new v rows (as cached), their scales | probabilities | warp
// maxima, denominators, outputs | scales of the warps' rows (compressed cache).  The fp32 new rows share the place of the warp outputs.
template <int D, int G, int MT> struct AttScratch {
    static constexpr int QS = 0, NEW = QS + G * D, NSC = NEW + MT * D, PW = NSC + 16, MM = PW + ST_NW * 64, ML = MM + ST_NW * 8, MO = ML + ST_NW * 8,
                         RAW = 2 * MT * D, SC = MO + (ST_NW * G * D > RAW ? ST_NW * G * D : RAW), FLOATS = SC + 2 * ST_KV_BLOCK;
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
    for (int j0 = c.tid; j0 < mine; j0 += U * ST_NT) {
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
        while (todo) {
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (todo >> i & 1u) t[i] = get2(at[i]);
#pragma unroll
            for (int i = 0; i < U; ++i)
                if ((todo >> i & 1u) && both(t[i], tag)) todo &= ~(1u << i);
            if (todo && !sp.again(c.abort(), p.spin_limit)) { ok = false; break; }
        }
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (all >> i & 1u) {
                const int j = j0 + i * ST_NT, kv = j - q_units;
                const float lo = packet_value(t[i].a), hi = packet_value(t[i].b);
                if (kv < 0) {
                    float *d = base + A::QS + (j / half) * D + (j & (half - 1));
                    d[0] = lo * p.q_scale;
                    d[half] = hi * p.q_scale;
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
    att.start(base + A::QS, c.lane);
    float *pw = base + A::PW + c.warp * 64;
    // (the new rows come last, by the last warp of the CTA that ends with them)
#pragma unroll 1
    for (int t = share.t0;; t += ST_KV_BLOCK) {
        const bool fresh = t >= share.t1;
        if (fresh && n_new == 0) break;
        const int n = fresh ? n_new : min(ST_KV_BLOCK, share.t1 - t);
        const int steps = (n + W::SP - 1) / W::SP, per_warp = (steps + ST_NW - 1) / ST_NW * W::SP;   // positions of a warp, whole steps
        int first = c.warp * per_warp, cnt = min(per_warp, n - first);
        const float *ksc = base + A::NSC, *vsc = ksc + 8;
        const unsigned char *at = reinterpret_cast<const unsigned char *>(base + A::NEW);
        if (fresh) {
            first = 0;
            cnt = c.warp == ST_NW - 1 ? n : 0;
        } else {
            if constexpr (Q8) {         // every warp fetches the scales of its own positions
                float *own = base + A::SC + c.warp * 16;
                const size_t row = (static_cast<size_t>(layer) * p.nkv + share.g) * p.max_context + t + first;
                if (c.lane < cnt) { own[c.lane] = __ldcg(p.k_scale + row + c.lane); own[8 + c.lane] = __ldcg(p.v_scale + row + c.lane); }
                __syncwarp();
                ksc = own;
                vsc = own + 8;
            }
            if (!chunk_wait(c, at)) { ok = false; break; }
        }
        if (cnt > 0) att.block(at, at + n * W::ROW, ksc, vsc, first, cnt, pw, c.lane);
        if (fresh) break;
        chunk_release(c);
    }
    att.leave(base + A::MM, base + A::ML, base + A::MO, c.warp, c.lane);
    if (!cta_vote(ok)) return false;
    // merge the warps and publish: one pair of dims per thread
    const size_t slot = static_cast<size_t>(share.tok) * c.sh().n_chunks + share.chunk;
#pragma unroll 1
    for (int j = c.tid; j < G * half; j += ST_NT) {
        const int h = j / half, d2 = j - h * half;
        float mw[ST_NW], mm = -INFINITY;
#pragma unroll
        for (int w = 0; w < ST_NW; ++w) { mw[w] = base[A::MM + w * 8 + h]; mm = fmaxf(mm, mw[w]); }
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int w = 0; w < ST_NW; ++w) {
            const float e = exp2_approx(mw[w] - mm);
            const float2 v = *reinterpret_cast<const float2 *>(base + A::MO + (w * G + h) * D + 2 * d2);
            a = fmaf(v.x, e, a);
            b = fmaf(v.y, e, b);
        }
        put2(p.part_ll + slot * p.qd + (share.g * G + h) * D + 2 * d2, a, b, tag);
    }
    if (c.tid < G) {                    // maximum and denominator of every head, one store
        float mm = -INFINITY, ll = 0.f;
#pragma unroll
        for (int w = 0; w < ST_NW; ++w) mm = fmaxf(mm, base[A::MM + w * 8 + c.tid]);
#pragma unroll
        for (int w = 0; w < ST_NW; ++w) ll = fmaf(base[A::ML + w * 8 + c.tid], exp2_approx(base[A::MM + w * 8 + c.tid] - mm), ll);
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
    const int lp = MT == 1 || n_chunks > 16 ? 32 : n_chunks > 8 ? 16 : 8, sub = c.lane & (lp - 1), per_warp = 32 / lp;
    bool ok = true;
#pragma unroll 1
    for (int it = c.warp * per_warp; it < n_pairs * m && ok; it += ST_NW * per_warp) {
        const int item = it + c.lane / lp;
        const bool on = item < n_pairs * m;
        const int tok = on ? item / n_pairs : 0, k_pair = on ? item - tok * n_pairs : 0, pr = a0 + k_pair, h = 2 * pr / p.D;
        float mx = -INFINITY, l = 0.f, a = 0.f, b = 0.f;      // of this lane's chunks
#pragma unroll 1
        for (int k0 = sub; k0 < n_chunks && on; k0 += lp * NJ) {
            Two st[NJ], ov[NJ];
            unsigned todo = 0;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                if (k0 + lp * j < n_chunks) todo |= 1u << j;
            const unsigned mine = todo;
            Spin sp;
            while (todo) {
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
                if (todo && !sp.again(c.abort(), p.spin_limit)) break;
            }
            if (todo) { ok = false; break; }
            float mn = mx;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                if (mine >> j & 1u) mn = fmaxf(mn, packet_value(st[j].a));
            const float f = mx == -INFINITY ? 0.f : exp2_approx(mx - mn);
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
        ok = __all_sync(0xffffffffu, ok);
        float mm = mx;
        for (int k = lp >> 1; k; k >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, k));
        const float f = mx == -INFINITY ? 0.f : exp2_approx(mx - mm);
        l *= f; a *= f; b *= f;
        for (int k = lp >> 1; k; k >>= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, k);
            a += __shfl_xor_sync(0xffffffffu, a, k);
            b += __shfl_xor_sync(0xffffffffu, b, k);
        }
        if (on && sub == 0) *reinterpret_cast<float2 *>(&c.sh().merged[tok][2 * k_pair]) = make_float2(a / l, b / l);
    }
    if (!cta_vote(ok)) return false;
    if constexpr (st_packets(MT)) {
        // a line is written by one instruction: every further write invalidates the pollers' copies of it (+ 1.5 us)
        const unsigned real_tag = tag ^ c.sh().odd;
#pragma unroll 1
        for (int i = c.tid; i < n_pairs * MT; i += ST_NT) {        // (unused tokens too: their slots keep up with the tags)
            const int tok = i / n_pairs, k = i - tok * n_pairs;
            const float2 v = tok < m ? *reinterpret_cast<const float2 *>(&c.sh().merged[tok][2 * k]) : make_float2(0.f, 0.f);
            put_raw2(p.ao_ll + (static_cast<size_t>(tok) * c.ncta + c.cta) * p.ao_line + 2 * k, pieces_packet(v.x, real_tag), pieces_packet(v.y, real_tag));
        }
    } else {
        const int stride = st_array_bytes(p.qd);
#pragma unroll 1
        for (int i = c.tid; i < 2 * n_pairs * m; i += ST_NT) {
            const int tok = i / (2 * n_pairs), k = i - tok * 2 * n_pairs;
            store_pieces<MT>(p.ao_vec, tok, 2 * a0 + k, stride, c.sh().merged[tok][k]);
        }
    }
    return true;
}

}  // namespace step
}  // namespace edgefm
