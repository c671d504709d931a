#define ST_TIGHT 1
#include "step_kernel.cuh"
namespace edgefm {
StepKernel step_tight_d64_m2(int G) { return ST_NS::kernel_for<64, false, 2>(G); }
}  // namespace edgefm
