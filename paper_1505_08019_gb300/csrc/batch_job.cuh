// batch_job.cuh -- which image of a grouped launch a CTA works on.
#pragma once

#include "passes.h"

namespace fft2d {

// Index of the job that owns this CTA.
template <class Table>
__device__ __forceinline__ int find_job(const Table &t)
{
    int lo = 0, hi = t.n - 1;
    const int b = (int)blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (t.job[mid].first_cta <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

}  // namespace fft2d
