// rb_scale.cuh -- power-of-two scaling of the reduced basis' rows and columns, for both precisions.
#pragma once

namespace fewsum {

constexpr int kRbMaxExp = 100;  // bound on the power-of-two scaling exponents (mixed)

// Exponent e with m 2^e in [2^14, 2^15) for m > 0 (0 for m = 0), clamped to +-kRbMaxExp.
__device__ __forceinline__ int scale_exp(float m)
{
    if (!(m > 0.0f)) return 0;
    const int e = 14 - (int)((__float_as_uint(m) >> 23) & 0xffu) + 127;
    return e > kRbMaxExp ? kRbMaxExp : (e < -kRbMaxExp ? -kRbMaxExp : e);
}

constexpr int kPlain = 10000;  // exponent of a row or column for the plain FP64 chain

// Exponent e with m 2^e in [1/2, 1) for m > 0 (0 for m = 0); kPlain outside 2^+-400.
__device__ __forceinline__ int scale_exp64(double m)
{
    if (m == 0.0) return 0;
    const int e = (int)((unsigned)__double2hiint(m) >> 20 & 0x7ffu);
    if (e < 1023 - 400 || e > 1023 + 400) return kPlain;
    return 1022 - e;
}

// |x| as an integer that orders as the magnitudes do, infinities and NaN above all numbers.
__device__ __forceinline__ unsigned long long mag(double x)
{
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

}  // namespace fewsum
