#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_kernel_q8_d128(int G) { return step::kernel_for<128, true>(G); }
}  // namespace edgefm
