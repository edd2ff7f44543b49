// Reciprocals and quotients without the division's length, from the hardware's approximations: FP64
// operations hold this part's scarce FP64 units for 65 clocks each, and a division takes about ten of them
// one after the other.  Compared with CUDA's own results over every exponent by tests/test_gpu_reciprocal.py.
#pragma once

#include <cuda_runtime.h>

namespace xk {

// 1 / x from the hardware's approximation (some 20 bits) by one third-order step, y (1 + e + e^2) with
// e = 1 - x y: the series of 1 / (1 - e).  Three dependent FP64 operations of 65 clocks each on this
// part, where a division takes about ten.  The division where the approximation's range ends (the
// exponent looked at as an integer).
__device__ __forceinline__ double reciprocal64(double x)
{
    const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    if (ex - 32u > 1984u) return 1.0 / x;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// 1 / x correctly rounded, without the division's length: reciprocal64 is within one unit in the last
// place, and from there y + y (1 - x y) rounds correctly (Markstein 1990) unless x's fraction is all
// ones.  That case, and exponents at which the residual may not be exact, take the division.
__device__ __forceinline__ double reciprocal_rn(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), ex = (hi >> 20) & 0x7ffu;
    if (ex - 64u > 1900u || ((hi & 0xfffffu) == 0xfffffu && __double2loint(x) == -1)) return 1.0 / x;
    const double y = reciprocal64(x);
    return fma(y, fma(-x, y, 1.0), y);
}

// x / d, correctly rounded, from rd = reciprocal_rn(d): the product q = x rd is within a unit of the
// quotient, and q + rd (x - q d) rounds correctly (Markstein 1990) while the residual is exact and the
// quotient a normal number, as it is for exponents of x and d within some 2^508 of one.  Three dependent
// FP64 operations where a division takes some ten.  Elsewhere the division itself (a d below 2^-1024 has
// an infinite reciprocal, and 0 x inf is no quotient); a zero x needs neither.
__device__ __forceinline__ double over(double x, double d, double rd)
{
    const unsigned hx = (unsigned)__double2hiint(x) & 0x7fffffffu, hd = (unsigned)__double2hiint(d) & 0x7fffffffu;
    const double q = x * rd;
    if ((hd >> 20) - 515u <= 1015u) {
        if ((hx >> 20) - 515u <= 1015u) return fma(fma(-q, d, x), rd, q);
        if ((hx | (unsigned)__double2loint(x)) == 0u) return q;
    }
    return x / d;
}

// 1 / x within one unit in the last place by two Newton-Raphson steps; the division where the
// approximation's range ends.
__device__ __forceinline__ double reciprocal_newton(double x)
{
    const double ax = fabs(x);
    if (!(ax > 1e-290 && ax < 1e290)) return 1.0 / x;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

// 1 / x in FP32 within one unit in the last place: the approximation and one Newton-Raphson step, the
// division unless that is a normal number (the approximation takes a subnormal x or result for zero).  The
// division everywhere cost 68 us instead of 63 for a leaf of 160 rows.
__device__ __forceinline__ float reciprocal32(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    const float z = fmaf(y, fmaf(-x, y, 1.0f), y);
    return (__float_as_uint(z) & 0x7fffffffu) - 0x00800000u < 0x7f000000u ? z : 1.0f / x;
}

}  // namespace xk
