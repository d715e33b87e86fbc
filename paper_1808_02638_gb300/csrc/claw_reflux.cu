// claw_reflux.cu -- the conservation fix's own launches (claw_reflux.cuh has the method) and the launch
// that averages the fine level onto the coarse one and applies the fix.
#include <cuda_runtime.h>

#include <algorithm>

#include "claw_average.cuh"
#include "claw_reflux.cuh"

namespace claw {
namespace {

constexpr int kThreads = 128;

template <int LIM> __global__ void __launch_bounds__(kThreads) reflux_kernel(const __grid_constant__ StepArgs A)
{
    refl::run_jobs<LIM, kThreads>(A, 0, gridDim.x);
}

// one thread per corrected coarse cell: its records in table order (deterministic sums)
__device__ __forceinline__ void apply_group(const RefluxRec* __restrict__ recs, int n, const int* __restrict__ group,
                                            int g, int ratio, const PatchDev* __restrict__ cp,
                                            const double* __restrict__ dt, const double* __restrict__ buf,
                                            double* __restrict__ qc)
{
    const int r0 = group[g], r1 = group[g + 1];
    const RefluxRec R0 = recs[r0];
    const PatchDev C = cp[R0.cbox];
    const double d = __ldg(dt + C.run) * C.dtscale;
    const double w = 1.0 / ((double)ratio * ratio);
    double corr[3] = {0.0, 0.0, 0.0};
    for (int r = r0; r < r1; ++r) {
        const RefluxRec R = recs[r];
        const double s = -R.side * d * (R.dir == 0 ? C.dxinv : C.dyinv);
        for (int m = 0; m < 3; ++m) {
            double fine = 0.0;
            for (int b = 0; b < ratio; ++b) fine += buf[3 * (n + r * ratio + b) + m];
            corr[m] = fma(s, fma(w, fine, buf[3 * r + m]), corr[m]);
        }
    }
    const int W = C.nx + 4;
    const long long WH = (long long)W * (C.ny + 4);
    const long long o = C.qoff + (long long)(R0.cj + 2) * W + (R0.ci + 2);
    for (int m = 0; m < 3; ++m) qc[o + m * WH] += corr[m];
}

// blocks [0, nb_avg) average (as average_kernel), the others correct: the fix touches coarse cells that
// the fine level does not cover, the average those that it does
__global__ void __launch_bounds__(kAverageThreads)
    average_reflux_kernel(const AvgRect* __restrict__ rects, int nrects, int nb_avg, int ratio,
                          const double* __restrict__ qf, const RefluxRec* __restrict__ recs, int n,
                          const int* __restrict__ group, int ng, const PatchDev* __restrict__ cp,
                          const double* __restrict__ dt, const double* __restrict__ buf, double* __restrict__ qc)
{
    if ((int)blockIdx.x < nb_avg) {
        average_block(rects, nrects, nb_avg, ratio, qf, qc);
        return;
    }
    const int g = ((int)blockIdx.x - nb_avg) * kAverageThreads + (int)threadIdx.x;
    if (g < ng) apply_group(recs, n, group, g, ratio, cp, dt, buf, qc);
}

}  // namespace

cudaError_t launch_reflux(const StepArgs& a, int limiter, cudaStream_t s)
{
    int n = 0;
    for (int j = 0; j < a.nreflux; ++j) n += refl::job_items(a.reflux[j]);
    if (n <= 0) return cudaSuccess;
    const int per = kThreads / refl::kLanes, grid = (n + per - 1) / per;
    switch (limiter) {
    case CLAW_LIM_NONE: reflux_kernel<CLAW_LIM_NONE><<<grid, kThreads, 0, s>>>(a); break;
    case CLAW_LIM_MINMOD: reflux_kernel<CLAW_LIM_MINMOD><<<grid, kThreads, 0, s>>>(a); break;
    case CLAW_LIM_SUPERBEE: reflux_kernel<CLAW_LIM_SUPERBEE><<<grid, kThreads, 0, s>>>(a); break;
    case CLAW_LIM_VANLEER: reflux_kernel<CLAW_LIM_VANLEER><<<grid, kThreads, 0, s>>>(a); break;
    case CLAW_LIM_MC: reflux_kernel<CLAW_LIM_MC><<<grid, kThreads, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_average_reflux(const AvgRect* r, int nrects, int max_cells, const double* qf, const RefluxRec* rec,
                                  int n, const int* group, int ngroups, int ratio, const PatchDev* cp,
                                  const double* dt, const double* buf, double* qc, cudaStream_t s)
{
    const int nb = average_blocks(nrects, max_cells), na = (ngroups + kAverageThreads - 1) / kAverageThreads;
    if (nb + na == 0) return cudaSuccess;
    average_reflux_kernel<<<nb + na, kAverageThreads, 0, s>>>(r, nrects, nb, ratio, qf, rec, n, group, ngroups, cp, dt,
                                                              buf, qc);
    return cudaGetLastError();
}

}  // namespace claw
