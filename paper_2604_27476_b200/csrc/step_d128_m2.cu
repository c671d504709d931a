#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_d128_m2(int G) { return step::kernel_for<128, false, 2>(G); }
}  // namespace edgefm
