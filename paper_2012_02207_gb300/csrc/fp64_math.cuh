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

// 1/sqrt(x) out of that range (zero for zero), by the library's functions
__device__ __noinline__ inline double inv_sqrt_slow(double x) { return x > 0.0 ? 1.0 / sqrt(x) : 0.0; }

__device__ __forceinline__ double inv_sqrt_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}

// mr = m / sqrt(x) and mr3 = m / sqrt(x)^3. The seed y (rsqrt.approx.ftz.f64,
// relative error below 2^-20, its low word zero, so y^2 is exact) leaves
// e = 1 - x y^2 with one rounding, and
//   x^(-1/2) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2 / 8 + O(e^3)),
//   1/x      = y^2 (1 + e + e^2 + O(e^3)),
// with e^3 below 2^-58. Both corrections are added to the leading term, so the
// results carry one or two roundings (two Newton steps from an FP32 seed took
// four more FP64 instructions, two of them conversions).
__device__ __forceinline__ void inv_powers(double x, double m, double& mr, double& mr3) {
    const double y = inv_sqrt_seed(x);
    const double y2 = y * y;
    const double e = fma(-x, y2, 1.0);
    const double w = e * fma(0.375, e, 0.5);
    const double my = m * y;
    mr = fma(my, w, my);
    mr3 = mr * fma(y2, fma(e, e, e), y2);
    if (!inv_in_range(x)) {
        const double rinv = inv_sqrt_slow(x);
        mr = m * rinv;
        mr3 = mr * rinv * rinv;
    }
}

// x^(-1/2) alone
__device__ __forceinline__ double inv_sqrt(double x) {
    const double y = inv_sqrt_seed(x);
    const double e = fma(-x, y * y, 1.0);
    return inv_in_range(x) ? fma(y, e * fma(0.375, e, 0.5), y) : inv_sqrt_slow(x);
}

}  // namespace gbfmm
