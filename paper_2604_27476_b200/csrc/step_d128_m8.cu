#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_d128_m8(int G) { return step::kernel_for<128, false, 8>(G); }
}  // namespace edgefm
