// Instantiations of the fused level-step for a uniform medium that take pulled ghosts.
#include "claw_step_uniform.cuh"

namespace claw {
StepKernel step_kernel_uniform_pull(int lim, int tx, int ty, int nt, int staging)
{
    return uniform_kernel_for<1>(lim, tx, ty, nt, staging);
}
}  // namespace claw
