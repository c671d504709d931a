#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_d64_m8(int G) { return step::kernel_for<64, false, 8>(G); }
}  // namespace edgefm
