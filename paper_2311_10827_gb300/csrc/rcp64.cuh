// The FP64 reciprocal of the step kernels.  Internal header.
#pragma once

#include <cuda_runtime.h>

namespace wblbm {

// 1/x to about one rounding: the hardware's 20-bit estimate r and one step of
// Householder's third-order iteration, e = 1 - x r, r (1 + e + e^2), whose
// error is e^3 < 2^-57.  x = rho tau_g, positive and of order one.
__device__ __forceinline__ double rcp64(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(fma(e, e, e), r, r);
}

}  // namespace wblbm
