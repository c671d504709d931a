#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_kernel_q8_d64(int G) { return step::kernel_for<64, true>(G); }
}  // namespace edgefm
