// The builds of the decode-step kernel and what the host has to know about them.
#include "step_attention.cuh"
#include "step_feed.cuh"

namespace edgefm {
StepKernel step_d64_m1(int G);
StepKernel step_d64_m2(int G);
StepKernel step_d64_m4(int G);
StepKernel step_d64_m8(int G);
StepKernel step_q8_d64_m1(int G);
StepKernel step_q8_d64_m8(int G);
StepKernel step_d128_m1(int G);
StepKernel step_d128_m2(int G);
StepKernel step_d128_m4(int G);
StepKernel step_d128_m8(int G);
StepKernel step_q8_d128_m1(int G);
StepKernel step_q8_d128_m8(int G);
StepKernel step_tight_d64_m1(int G);
StepKernel step_tight_d64_m2(int G);
StepKernel step_tight_d64_m4(int G);
StepKernel step_tight_q8_d64_m1(int G);
StepKernel step_tight_d128_m1(int G);
StepKernel step_tight_d128_m2(int G);
StepKernel step_tight_d128_m4(int G);
StepKernel step_tight_q8_d128_m1(int G);

StepKernel step_kernel_for(int D, int G, bool kv8, int mt, bool tight) {
    if (tight) {
        if (kv8) return mt != 1 ? nullptr : D == 64 ? step_tight_q8_d64_m1(G) : step_tight_q8_d128_m1(G);
        switch (mt) {
            case 1: return D == 64 ? step_tight_d64_m1(G) : step_tight_d128_m1(G);
            case 2: return D == 64 ? step_tight_d64_m2(G) : step_tight_d128_m2(G);
            case 4: return D == 64 ? step_tight_d64_m4(G) : step_tight_d128_m4(G);
            default: return nullptr;
        }
    }
    if (kv8) {
        if (mt == 1) return D == 64 ? step_q8_d64_m1(G) : step_q8_d128_m1(G);
        if (mt == 8) return D == 64 ? step_q8_d64_m8(G) : step_q8_d128_m8(G);
        return nullptr;
    }
    switch (mt) {
        case 1: return D == 64 ? step_d64_m1(G) : step_d128_m1(G);
        case 2: return D == 64 ? step_d64_m2(G) : step_d128_m2(G);
        case 4: return D == 64 ? step_d64_m4(G) : step_d128_m4(G);
        case 8: return D == 64 ? step_d64_m8(G) : step_d128_m8(G);
        default: return nullptr;
    }
}
int step_shared_bytes(int mt) {
    using namespace step;
    return mt == 1 ? st_shared_bytes<1>() : mt == 2 ? st_shared_bytes<2>() : mt == 4 ? st_shared_bytes<4>() : st_shared_bytes<8>();
}
template <int D, int MT> static int scratch(int G) {
    using namespace step;
    switch (G) {
        case 1: return AttScratch<D, 1, MT>::FLOATS;
        case 2: return AttScratch<D, 2, MT>::FLOATS;
        case 3: return AttScratch<D, 3, MT>::FLOATS;
        case 4: return AttScratch<D, 4, MT>::FLOATS;
        case 5: return AttScratch<D, 5, MT>::FLOATS;
        case 6: return AttScratch<D, 6, MT>::FLOATS;
        case 7: return AttScratch<D, 7, MT>::FLOATS;
        default: return AttScratch<D, 8, MT>::FLOATS;
    }
}
template <int D> static int scratch_of(int G, int mt) { return mt == 1 ? scratch<D, 1>(G) : mt == 2 ? scratch<D, 2>(G) : mt == 4 ? scratch<D, 4>(G) : scratch<D, 8>(G); }
int step_scratch_floats(int D, int G, int mt) { return D == 64 ? scratch_of<64>(G, mt) : scratch_of<128>(G, mt); }
int step_chunks(const StepLaunch &sl, int op, int cta, unsigned *out, int capacity) {
    const StepParams &p = sl.p;
    const int units = step::op_units(p, op, p.V);
    int at = 0;
    for (int u = st_first(units, cta, sl.grid), u1 = st_first(units, cta + 1, sl.grid), n; u < u1; u += n) {
        n = step::tile_units(p, op, u, u1);
        for (int s = 0; s < p.cols[op].segs; ++s, ++at) {
            if (at >= capacity) continue;
            const uint4 e = step::chunk_entry(p, op, u, n, s);
            const unsigned v[6] = {e.x, e.y, e.z, e.w, static_cast<unsigned>(u), static_cast<unsigned>(n)};
            std::copy(v, v + 6, out + 6 * static_cast<size_t>(at));
        }
    }
    return at;
}
}  // namespace edgefm
