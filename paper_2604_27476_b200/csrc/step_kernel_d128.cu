#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_kernel_d128(int G) { return step::kernel_for<128, false>(G); }
}  // namespace edgefm
