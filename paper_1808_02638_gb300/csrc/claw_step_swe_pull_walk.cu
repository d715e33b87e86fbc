// Shallow-water level-step kernels: pulled ghosts, column walks.
#include "claw_step_swe.cuh"

namespace claw {

StepKernel step_kernel_swe_pull_walk(int lim, int tx, int ty, int nt, int staging)
{
    return swe_for<true, true>(lim, tx, ty, nt, staging);
}

}  // namespace claw
