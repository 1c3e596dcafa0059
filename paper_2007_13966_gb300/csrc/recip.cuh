// The FP64 reciprocal of the EOS, the subdomain factorisation and the coarse pivots.
#pragma once

#include "common.cuh"

namespace ras {

// 1 / x by one step of the hyperpower iteration of order three (M. Altman, 1960),
// y (1 + e + e^2) with e = 1 - x y, from the FP32 reciprocal y of x rounded to FP32:
// |e| < 2^-22, so that e^3 is below 2^-66 of the result and its error that of the last
// rounding. Where x lies in FP32's normal range with room (1e-36 to 1e36); the division
// otherwise. Three dependent operations of the FP64 pipe (2 per cycle and SM, ~64 cycles
// each) and two conversions, where a division takes about ten (~440 cycles).
__device__ __forceinline__ double recip64(double x) {
    const double ax = fabs(x);
    if (!(ax > 1e-36 && ax < 1e36)) return 1.0 / x;
    const double y = (double)__frcp_rn((float)x);
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

}  // namespace ras
