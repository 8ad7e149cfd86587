// gt_math.h -- arithmetic that the host compiler takes too, so that it can be
// compared with the C library's without a GPU.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define GT_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define GT_HOST_DEVICE inline
#endif

namespace gt {

// n / d, correctly rounded, for a divisor known in advance with r = 1/d
// rounded: the first residual step makes the quotient faithful, the second
// rounds it correctly (Markstein, IBM J. Res. Dev. 34, 111, 1990), while r,
// the quotient and the residuals are normal numbers.
GT_HOST_DEVICE float div_known32(float n, float d, float r)
{
    float q = n * r;
    q = fmaf(fmaf(-q, d, n), r, q);
    return fmaf(fmaf(-q, d, n), r, q);
}

}  // namespace gt
