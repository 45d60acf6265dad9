// Square roots in FP64 with few FP64 operations (GB300 retires 2 FP64 lanes
// per clock and SM; the library's root and quotient take three times as many).
//
// 1/sqrt(r) from an FP32 seed y by one step of Householder's method of third
// order: with e = 1 - r y^2, 1/sqrt(r) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8
// + O(e^3)).  The seed's relative error is below 2^-21, so |e| < 2^-20 and the
// rest, 5/16 e^3, is below 2^-61.  What counts is rounding: r y is rounded (at
// most 2^-53, halved in the result) and the result (2^-53): 1.5 x 2^-53 in all,
// where the quotient by a rounded root has 2^-52.
#pragma once

#include <cuda_runtime.h>

namespace pmroot {

// The range of the FP32 seed, with room; outside it the library's functions.
constexpr double LO = 1e-30, HI = 1e30;

// The FP64 value of a normal FP32 one by integer operations (the conversion
// takes a slot of the FP64 pipe).
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f);   // f > 0
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}
// 1/sqrt(r), r known to FP32 as rf (relative error below 2^-22).
__device__ __forceinline__ double inv_sqrt(double r, float rf) {
    if (!(rf > (float)LO && rf < (float)HI)) return 1.0 / sqrt(r);
    const double y = widen(rsqrtf(rf));
    const double e = fma(-(r * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
// R = sqrt(r) and inv = 1/R (0 for 0).  R from inv by one Newton step on the
// residual r - R^2, which an FMA gives exactly: what is left beside the last
// rounding is below 2^-100, so R is the correctly rounded root but for
// arguments whose root lies within 2^-47 units of a rounding boundary.
__device__ __forceinline__ void root_inv(double r, double &R, double &inv) {
    if (!(r > LO && r < HI)) {
        R = __dsqrt_rn(r);
        inv = R > 0 ? 1.0 / R : 0.0;
        return;
    }
    const double y = (double)rsqrtf((float)r);
    const double e = fma(-(r * y), y, 1.0);
    inv = fma(y * e, fma(0.375, e, 0.5), y);
    R = r * inv;
    R = fma(0.5 * inv, fma(-R, R, r), R);
}

}  // namespace pmroot
