#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_kernel_d64(int G) { return step::kernel_for<64, false>(G); }
int step_shared_bytes() { return step::ST_SHARED_BYTES; }
int step_scratch_floats(int D, int G) {
    using step::AttScratch;
    // (linear in G)
    return D == 64 ? AttScratch<64, 1>::FLOATS + (G - 1) * (AttScratch<64, 2>::FLOATS - AttScratch<64, 1>::FLOATS)
                   : AttScratch<128, 1>::FLOATS + (G - 1) * (AttScratch<128, 2>::FLOATS - AttScratch<128, 1>::FLOATS);
}
}  // namespace edgefm
