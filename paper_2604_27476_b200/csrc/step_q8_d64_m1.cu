#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_q8_d64_m1(int G) { return step::kernel_for<64, true, 1>(G); }
}  // namespace edgefm
