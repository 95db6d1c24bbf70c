// newton.h -- reciprocal and reciprocal square root in FP64 by Newton's iteration
// from a seed of FP32 accuracy (for host and device).  The residual of the last step
// is formed with fused multiply-adds, free of rounding but for the residual's own, so
// the result is the exact value rounded once, but within 2^-30 or so of a tie.
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define RELOC_HD __host__ __device__ __forceinline__
#else
#define RELOC_HD inline
#endif

namespace reloc {

// 1 / x from a seed r.
RELOC_HD double newton_recip(double x, double r)
{
    r = fma(fma(-x, r, 1.0), r, r);
    return fma(fma(-x, r, 1.0), r, r);
}

// 1 / sqrt(x) from a seed r.  The last step's product x r is taken with its rounding
// error: without it the result is up to 0.98 ulp off, so 0.50.
RELOC_HD double newton_rsqrt(double x, double r)
{
    r = fma(fma(-x * r, r, 1.0), 0.5 * r, r);
    const double y = x * r, d = fma(x, r, -y);
    return fma(fma(-d, r, fma(-y, r, 1.0)), 0.5 * r, r);
}

}  // namespace reloc
