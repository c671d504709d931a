#define ST_TIGHT 1
#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_tight_d128_m4(int G) { return ST_NS::kernel_for<128, false, 4>(G); }
}  // namespace edgefm
