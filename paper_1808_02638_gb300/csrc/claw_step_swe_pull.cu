// Shallow-water level-step kernels: pulled ghosts, striding CTAs.
#include "claw_step_swe.cuh"

namespace claw {

StepKernel step_kernel_swe_pull(int lim, int tx, int ty, int nt, int staging)
{
    return swe_for<true, false>(lim, tx, ty, nt, staging);
}

}  // namespace claw
