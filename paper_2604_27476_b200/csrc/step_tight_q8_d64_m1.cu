#define ST_TIGHT 1
#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_tight_q8_d64_m1(int G) { return ST_NS::kernel_for<64, true, 1>(G); }
}  // namespace edgefm
