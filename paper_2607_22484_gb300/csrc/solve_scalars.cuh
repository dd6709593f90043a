// Device scalars of a solve that more than one kernel computes.
#pragma once

#include <cuda_runtime.h>

namespace svt {

namespace {

// alpha = 2^e with e = round(log2 ||A||_F) (1 for a zero matrix): dividing by it is exact.
__device__ __forceinline__ double pow2_alpha(double nrm2)
{
    if (!(nrm2 > 0.0) || !isfinite(nrm2))
        return 1.0;
    int e;
    double f = frexp(sqrt(nrm2), &e);  // sqrt = f 2^e, f in [0.5, 1)
    if (f < 0.70710678118654752)
        e -= 1;
    return ldexp(1.0, e);
}

// theta = src^(1/4) (quarter) or src^(1/2). Roots and products in place of pow: FP64 runs at
// 2 lanes a cycle and SM, and a first step waits for its scales.
__device__ __forceinline__ double root_theta(double src, bool quarter)
{
    const double r = sqrt(src);
    return quarter ? sqrt(r) : r;
}

// x^e for small e >= 0.
__device__ __forceinline__ double int_pow(double x, int e)
{
    double p = 1.0;
    for (int i = 0; i < e; ++i)
        p *= x;
    return p;
}

} // namespace

} // namespace svt
