// Step kernel for four CTAs an SM (one translation unit each, compiled in parallel).
#include "pat_step.cuh"

namespace pat {
StepKernel step_kernel_r4() { return step_kernel<4>; }
}  // namespace pat
