// Exact-digit arithmetic of the FP64 products (see hps_digit.cu): the split of
// FP64 entries into eight balanced base-256 digits as FP16 integers, and the
// rounding of a fixed-point sum with its scale.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace hps {
namespace {

constexpr int DG_S = 8;      // digits of an operand
constexpr int E_MIN = 1;     // scale exponent of a row or column of zeros (exp_of: subnormal entries count as zero)
constexpr int E_BAD = 2047;  // an infinity or NaN (exp_all: or a subnormal) in the row or column: its scale is then kept as E_NAN
constexpr int E_NAN = 1 << 20;

__device__ __forceinline__ int exp_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int exp_all(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x);
    return exp_of(x) == 0 && ((hi << 1) | (uint32_t)__double2loint(x)) != 0 ? E_BAD : exp_of(x);
}

// Bits 0 .. 3: the entry is within 2^-reach of the scale; 4 .. 7: it is not zero.
__device__ __forceinline__ unsigned char reach4(const double (&x)[4], int E, int reach)
{
    uint32_t m = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int e = (int)(((uint32_t)__double2hiint(x[u]) >> 20) & 0x7ffu);
        m |= (uint32_t)(e >= max(E - reach, 1)) << u | (uint32_t)(e != 0) << (4 + u);
    }
    return (unsigned char)m;
}
// Digits of four entries under the scale exponent E: digit s of entries 0, 1
// as FP16 pairs in d[s][0], of entries 2, 3 in d[s][1].
__device__ __forceinline__ void split4(const double (&x)[4], int E, uint32_t (&d)[DG_S][2])
{
    uint32_t w[4][2];
    __half2 sg[2], off[2], off0[2];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint32_t hi = (uint32_t)__double2hiint(x[u]), lo = (uint32_t)__double2loint(x[u]);
        const int e = (int)((hi >> 20) & 0x7ffu);
        const int sh = e ? min(E - e, 63) : 63;   // zero (and subnormal) entries: all digits zero
        const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
        const uint64_t m = ((((uint64_t)mh << 32) | lo) << 9) >> sh;
        const uint64_t b = m + 0x0080808080808080ull;   // balanced digits: byte - 128 below the leading one
        w[u][0] = (uint32_t)b;
        w[u][1] = (uint32_t)(b >> 32);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // +-1 of the two entries, and the biases of 1024 + byte that belong to them
        const uint32_t h0 = (uint32_t)__double2hiint(x[2 * h]), h1 = (uint32_t)__double2hiint(x[2 * h + 1]);
        const uint32_t sb = ((h0 >> 16) & 0x8000u) | (h1 & 0x80000000u);
        const uint32_t one = 0x3C003C00u ^ sb, o1152 = 0xE480E480u ^ sb, o1024 = 0xE400E400u ^ sb;
        sg[h] = *reinterpret_cast<const __half2*>(&one);
        off[h] = *reinterpret_cast<const __half2*>(&o1152);
        off0[h] = *reinterpret_cast<const __half2*>(&o1024);
    }
#pragma unroll
    for (int s = 0; s < DG_S; ++s) {
        const int byte = 7 - s;   // plane 0 holds the leading digit
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t a = w[2 * h][byte >> 2], b = w[2 * h + 1][byte >> 2];
            uint32_t v = __byte_perm(a, b, (uint32_t)(byte & 3) | ((uint32_t)(4 + (byte & 3)) << 8));
            v = (v & 0x00FF00FFu) | 0x64006400u;   // FP16 1024 + byte
            const __half2 v2 = __hfma2(*reinterpret_cast<const __half2*>(&v), sg[h], s == 0 ? off0[h] : off[h]);
            d[s][h] = *reinterpret_cast<const uint32_t*>(&v2);
        }
    }
}

// V 2^-57 of the scales, rounded once to FP64.  E: biased exponents of the two
// scales, less 1016 (a unit of 2^-(57 + j) takes j more off).  eb_out outside
// 0 .. 2045 asks for a plain sum instead: a result outside the normal range, or
// of a row or column of scale E_NAN.  No branch, so that several overlap.
__device__ __forceinline__ double round_fixed(long long V, int E, int& eb_out)
{
    const int sm = (int)(V >> 63);
    uint64_t u = (uint64_t)((V ^ (long long)sm) - (long long)sm);
    const int lz = __clzll((long long)u);              // 1 .. 63, 64 for zero
    u <<= (lz - 1) & 63;
    u += 512;                                          // the leading bit is bit 62: 53 bits stay
    int eb = E - lz;
    uint64_t r = (u >> 10) + ((uint64_t)(uint32_t)eb << 52);
    r |= (uint64_t)((uint32_t)sm & 0x80000000u) << 32;
    const bool zero = lz == 64 && E < (1 << 19);
    eb_out = zero ? 0 : lz == 64 ? 4096 : eb;
    return __longlong_as_double(zero ? 0ll : (long long)r);
}

}  // namespace
}  // namespace hps
