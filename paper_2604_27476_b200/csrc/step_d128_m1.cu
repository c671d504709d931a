#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_d128_m1(int G) { return step::kernel_for<128, false, 1>(G); }
}  // namespace edgefm
