// Instantiations of the fused level-step for a uniform medium (rho0, K0).
#include "claw_step_uniform.cuh"

namespace claw {
StepKernel step_kernel_uniform(int lim, int tx, int ty, int nt, int staging)
{
    return uniform_kernel_for<0>(lim, tx, ty, nt, staging);
}
}  // namespace claw
