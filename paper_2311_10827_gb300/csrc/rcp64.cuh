// The FP64 reciprocal and the relaxation of a population in the step kernels.
// Internal header.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace wblbm {

// 1/x: the hardware's estimate r and one step of Householder's third-order
// iteration, e = 1 - x r, r (1 + e + e^2), whose error is e^3.  An estimate good to
// 2^-19 leaves 1/16 of an ulp beside the final rounding's half.  For every
// positive or negative x for which x and 1/x are normal numbers (that is any
// density and relaxation time of a run); where the estimate is infinite or zero
// (x zero, subnormal, infinite or at least 2^1022) it is the result, which for
// zeros, infinities and NaN is the divide's.  The estimate's exponent is tested as an
// integer: the FP64 pipe, which bounds the kernels that use this, gets three
// operations.
__device__ __forceinline__ double rcp64(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    const double y = fma(fma(e, e, e), r, r);
    const unsigned k = ((unsigned)__double2hiint(r) >> 20) & 0x7ffu;
    return k - 1u < 0x7feu ? y : r;
}

// x relaxed by a rate r plus s, omr = 1 - r.  For r >= 1/2, 1 - r is exact and x (1 - r) + s
// one operation.  Below (tau > 2) it is rounded, and every population would
// relax by up to 2^-54 more or less than the r that the equilibrium part is
// multiplied by: a drift of the sums that should stay (phi, momentum) that
// grows with every step, where independent roundings average out.  There (INC)
// the population is moved by its increment -r x + s, one operation more.  A
// run's parameters choose (StepParams::incr), not a node's rate: warps on an
// interface would run both forms (64^3 312 us per step against 248).
template <bool INC>
__device__ __forceinline__ double relax64(double x, double r, double omr, double s)
{
    return INC ? x + fma(-r, x, s) : fma(omr, x, s);
}

}  // namespace wblbm
