#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_d64_m2(int G) { return step::kernel_for<64, false, 2>(G); }
}  // namespace edgefm
