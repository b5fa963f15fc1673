// Step kernel for three CTAs an SM (one translation unit each, compiled in parallel).
#include "pat_step.cuh"

namespace pat {
StepKernel step_kernel_r3() { return step_kernel<3>; }
}  // namespace pat
