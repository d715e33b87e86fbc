// Shallow-water level-step kernels: filled ghosts, striding CTAs.
#include "claw_step_swe.cuh"

namespace claw {

StepKernel step_kernel_swe(int lim, int tx, int ty, int nt, int staging)
{
    return swe_for<false, false>(lim, tx, ty, nt, staging);
}

}  // namespace claw
