// FP64 1/x and 1/sqrt(x) from the hardware's approximations, in fewer instructions of the
// FP64 unit than the divide and rsqrt take.
#pragma once

namespace fil {

// 1/x by Newton's iteration y += y (1 - x y) from the hardware's seed (about
// 2^-20): two steps, each one fused residual and one fused update, leave an
// error of rounding size. The seed flushes what 1/x or x would make subnormal,
// so those, infinities and NaN divide.
__device__ __forceinline__ double recip(double x) {
    const int e = (__double2hiint(x) >> 20) & 0x7ff;
    if (e < 2 || e > 2044) return 1.0 / x;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

// 1/sqrt(x) for normal x > 0: the hardware's approximation (PTX
// rsqrt.approx.ftz.f64, ~20 bits) and one step of the third-order iteration
//   y <- y + y e (1/2 + 3/8 e),  e = 1 - x y^2
// (the series of (1 - e)^{-1/2}), whose next term, 5/16 e^3, is below 2^-57.
__device__ __forceinline__ double rsqrt_iter(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    return fma(fma(0.375, e, 0.5), y * e, y);
}

}  // namespace fil
