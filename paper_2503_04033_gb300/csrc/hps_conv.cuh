#pragma once

#include <cuda_runtime.h>

namespace hps {
namespace {

// Conversions between FP64 and FP32 on the integer pipe (on GB300 the FP64
// pipe that executes the conversion instructions is the residual's and the
// refinement update's bottleneck).  Both follow the IEEE-754 binary64 /
// binary32 encodings; anything outside the normal range goes to the hardware
// conversion.  hps_selftest_conversions checks them bit for bit against it.
//
// double -> float, round to nearest even: the 52-bit significand is rounded
// to 23 bits by adding 0x0FFFFFFF plus the kept part's last bit before the
// 29-bit shift (a carry into the exponent is the correct result, up to
// infinity), and the exponent is rebiased from 1023 to 127.
__device__ __forceinline__ float d2f_rn(double x)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const unsigned long long a = u & 0x7FFFFFFFFFFFFFFFull;
    const unsigned e = (unsigned)(a >> 52);
    if (e - 897u > 253u) return __double2float_rn(x);   // zero, float subnormal or overflow, inf, NaN
    const unsigned long long r = (a + 0x0FFFFFFFull + ((a >> 29) & 1ull)) >> 29;
    const unsigned f = (unsigned)(r - (896ull << 23)) | (unsigned)((u >> 32) & 0x80000000u);
    return __uint_as_float(f);
}

// float -> double (exact): the significand moves up 29 bits and the exponent
// is rebiased from 127 to 1023; zero keeps its sign.
__device__ __forceinline__ double f2d(float x)
{
    const unsigned u = __float_as_uint(x);
    const unsigned e = (u >> 23) & 0xFFu;
    const unsigned long long sgn = (unsigned long long)(u >> 31) << 63;
    if (e - 1u > 253u) {
        if ((u << 1) == 0u) return __longlong_as_double((long long)sgn);
        return (double)x;                                  // subnormal, inf, NaN
    }
    return __longlong_as_double((long long)(((unsigned long long)(u & 0x7FFFFFFFu) << 29) + (896ull << 52) | sgn));
}

}  // namespace
}  // namespace hps
