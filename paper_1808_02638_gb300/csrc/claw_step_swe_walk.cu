// Shallow-water level-step kernels: filled ghosts, column walks.
#include "claw_step_swe.cuh"

namespace claw {

StepKernel step_kernel_swe_walk(int lim, int tx, int ty, int nt, int staging)
{
    return swe_for<false, true>(lim, tx, ty, nt, staging);
}

}  // namespace claw
