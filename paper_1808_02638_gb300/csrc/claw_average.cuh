// claw_average.cuh -- averaging of a fine level onto the coarse one ("updating", Sec. 2.2-2.3).
#pragma once

#include <algorithm>

#include "claw_internal.h"

namespace claw {

// Block b of a launch takes chunk b / nrects of rectangle b % nrects, a thread per (coarse cell,
// component).  One block per rectangle left most of the chip idle and looped over its largest with one
// dependent chain of loads and sums a thread at a time: 8 us for 169 rectangles of up to 256 cells.
constexpr int kAverageThreads = 128;

// chunks a rectangle is split into, for rectangles of up to max_cells coarse cells
inline int average_chunks(int max_cells)
{
    return std::max(1, std::min(64, (3 * max_cells + kAverageThreads - 1) / kAverageThreads));
}
inline int average_blocks(int nrects, int max_cells) { return nrects <= 0 ? 0 : nrects * average_chunks(max_cells); }

// the r x r children are summed row by row and divided by r^2 (an exact product for r = 2, 4), all of
// them loaded before the first sum
template <int RATIO>
__device__ __forceinline__ double mean_of(const double* __restrict__ f, int pitch)
{
    double v[RATIO * RATIO];
#pragma unroll
    for (int b = 0; b < RATIO; ++b)
#pragma unroll
        for (int a = 0; a < RATIO; ++a) v[b * RATIO + a] = f[(long long)b * pitch + a];
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < RATIO * RATIO; ++k) s += v[k];
    return s * (1.0 / (RATIO * RATIO));
}

__device__ __forceinline__ void average_block(const AvgRect* __restrict__ rects, int nrects, int nblocks, int ratio,
                                              const double* __restrict__ qf, double* __restrict__ qc)
{
    const int chunk = (int)blockIdx.x / nrects, chunks = nblocks / nrects;
    const AvgRect R = rects[(int)blockIdx.x - chunk * nrects];
    const int cells = R.w * R.h;
    for (int k = chunk * kAverageThreads + (int)threadIdx.x; k < 3 * cells; k += chunks * kAverageThreads) {
        const int m = k / cells, e = k - m * cells;
        const int y = e / R.w, x = e - y * R.w;
        const double* f = qf + R.fsrc + m * R.fplane + (long long)y * ratio * R.fpitch + (long long)x * ratio;
        double v;
        if (ratio == 2) v = mean_of<2>(f, R.fpitch);
        else if (ratio == 4) v = mean_of<4>(f, R.fpitch);
        else {
            v = 0.0;
            for (int b = 0; b < ratio; ++b)
                for (int a = 0; a < ratio; ++a) v += f[(long long)b * R.fpitch + a];
            v /= (double)(ratio * ratio);
        }
        qc[R.cdst + m * R.cplane + (long long)y * R.cpitch + x] = v;
    }
}

}  // namespace claw
