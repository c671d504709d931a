#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_d128_m4(int G) { return step::kernel_for<128, false, 4>(G); }
}  // namespace edgefm
