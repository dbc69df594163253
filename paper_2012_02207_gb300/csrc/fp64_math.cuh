// Powers of 1/r in FP64 for pair sums, in as few FP64 instructions as possible:
// GB300 runs an FP64 instruction of a warp for 64 cycles of its scheduler.
#pragma once

#include <cuda_runtime.h>

namespace gbfmm {

// x within [2^-999, 2^993): neither the seed nor the correction under- or
// overflows (an integer test: an FP64 comparison would cost an FP64 instruction)
__device__ __forceinline__ bool inv_in_range(double x) {
    return (unsigned)__double2hiint(x) - 0x01800000u < 0x7e000000u - 0x01800000u;
}

// mr = m / sqrt(x) and mr3 = m / sqrt(x)^3. The seed y (rsqrt.approx.ftz.f64,
// relative error below 2^-20, its low word zero, so y^2 is exact) leaves
// e = 1 - x y^2 with one rounding, and
//   x^(-1/2) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2 / 8 + O(e^3)),
//   1/x      = y^2 (1 + e + e^2 + O(e^3)),
// with e^3 below 2^-58. Both corrections are added to the leading term, so the
// results carry one or two roundings (the earlier two Newton steps from an FP32
// seed took four more FP64 instructions, two of them conversions). Zero gives
// zero; other values out of range take the library's division and square root.
__device__ __forceinline__ void inv_powers(double x, double m, double& mr, double& mr3) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double y2 = y * y;
    const double e = fma(-x, y2, 1.0);
    const double w = e * fma(0.375, e, 0.5);
    const double my = m * y;
    mr = fma(my, w, my);
    mr3 = mr * fma(y2, fma(e, e, e), y2);
    if (!inv_in_range(x)) {
        const double rinv = x > 0.0 ? 1.0 / sqrt(x) : 0.0;
        mr = m * rinv;
        mr3 = mr * rinv * rinv;
    }
}

}  // namespace gbfmm
