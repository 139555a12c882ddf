// 1/sqrt(d) in FP64 from CUDA's FP32 rsqrtf, for the pivots of the Cholesky kernels.
#pragma once

#include <math.h>

namespace tsvd {

// For finite d > 0: FP32 estimate of the scaled value, two Newton steps y <- y (3 - d y^2) / 2
// in FP64 (22 -> 43 -> beyond 53 bits; the last step's roundings leave 2 ulp at most), rescaled.
__device__ inline double rsqrt_fp64(double d) {
    const int e = ilogb(d) & ~1;  // even exponent: d = dd 2^e, dd in [1, 4)
    const double dd = scalbn(d, -e);
    double y = (double)rsqrtf((float)dd);
    y = y * fma(-0.5 * dd, y * y, 1.5);
    y = y * fma(-0.5 * dd, y * y, 1.5);
    return scalbn(y, -e / 2);
}

// The same with a short chain on the FP64 pipe, for a finite d > 0: one step of third order, the
// binomial series of (1 - e)^(-1/2) to its second term (Householder's iteration for y^-2 = d).
//   d is scaled by an even power of two to [1, 4); the scaling and both conversions are by bits.
//   y = rsqrtf of its leading 24 bits: relative error below 2^-21.5 (2 ulp of FP32, and 2^-24
//   for the bits left out), and y^2 is exact.
//   e = 1 - d y^2, |e| < 2^-20.5, rounded to 2^-73;
//   d^(-1/2) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + 5 e^3/16 + ..): what is left out is
//   below 2^-63, so the one rounding of the last fma counts: 0.51 ulp.
__device__ inline double rsqrt_fp64_short(double d) {
    const int hi = __double2hiint(d), lo = __double2loint(d);
    const int ex = ((hi >> 20) - 1023) & ~1;
    if ((hi >> 20) == 0) return rsqrt_fp64(d);  // subnormal
    const int h = hi - (ex << 20);  // exponent field 1023 or 1024
    const double dd = __hiloint2double(h, lo);
    const float f = __int_as_float(((h >> 20) - 896) << 23 | (h & 0xFFFFF) << 3 | (int)((unsigned)lo >> 29));
    const int yb = __float_as_int(rsqrtf(f));  // in (1/2, 1]
    const double y = __hiloint2double((yb >> 3) + (896 << 20), yb << 29);
    const double e = fma(-dd, y * y, 1.0);
    const double z = fma(y * e, fma(e, 0.375, 0.5), y);
    return __hiloint2double(__double2hiint(z) - ((ex >> 1) << 20), __double2loint(z));
}

}  // namespace tsvd
