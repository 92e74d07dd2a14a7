// near64.cuh -- FP64 pieces of the plain form's near field shared by near64.cu (uniform tree) and adaptive.cu.
#pragma once

#include "fmm_internal.cuh"

namespace fmm {

// F(x) for 0 <= x < N64_XCUT: the row from the bit pattern of x (integer operations), then one subtraction and six
// multiply-adds.
__device__ __forceinline__ int blob_row(double x)
{
    const int hi = __double2hiint(x);
    const int e = (hi >> 20) - 1023;
    return e >= -4 ? ((hi & 0xfffff) | 0x100000) >> (16 - e) : 0;
}
__device__ __forceinline__ double blob_poly(const double2 *__restrict__ tab, int i, double x)
{
    const double2 c01 = __ldg(tab + 4 * i), c23 = __ldg(tab + 4 * i + 1), c45 = __ldg(tab + 4 * i + 2),
                  c6c = __ldg(tab + 4 * i + 3);
    const double t = x - c6c.y;
    double f = fma(c6c.x, t, c45.y);
    f = fma(f, t, c45.x);
    f = fma(f, t, c23.y);
    f = fma(f, t, c23.x);
    f = fma(f, t, c01.y);
    return fma(f, t, c01.x);
}

// 1 / x to FP64 rounding for a normal x > 0: the SFU's seed (relative error below 2^-20) and one Newton step of third
// order, y (1 + e + e^2) with e = 1 - x y.
__device__ __forceinline__ double recip64(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

}  // namespace fmm
