#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_d64_m4(int G) { return step::kernel_for<64, false, 4>(G); }
}  // namespace edgefm
