// Squared distances of the FP64 and FP64X phase-2 scans on the integer pipe.
//
// GB300 runs FP64 arithmetic at 2 operations per clock per SM, so that the two operations of
// dx^2 + dy^2 cost a clock; the integer steps here are about 45 of an SM's 128 issue slots a
// clock. 16,384 x 262,144 with FP64X: 31.9 -> 27.1 ms (2 FP64 operations a pair instead of 4; now
// 78 % of the issue slots). The differences dx and dy stay FP64 subtractions. Their significands
// are squared to the high word of the 128-bit product, aligned, added and normalised: the sum is
// exact to about 2^-59 relative, where the FP64 form rounds it to 2^-52.
#pragma once

#include <cstdint>

#include "aidw_internal.cuh"

namespace aidw {

// A positive value m 2^(e - 63), m in [2^63, 2^64).
struct NormU64 {
    int e;
    unsigned long long m;
};

// x > 0, normal; +inf and NaN have e = 1024.
__device__ __forceinline__ NormU64 norm_of(double x)
{
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
    return {static_cast<int>(b >> 52) - 1023, (1ull << 63) | (b << 11)};
}

// dx^2 + dy^2, at least kEpsF64 = 2^-1022 (an exact coincidence gives exactly that). e > 1023 for
// an infinite or NaN difference (a padding point, a non-finite query) and where the sum would
// overflow a double.
__device__ __forceinline__ NormU64 sum_of_squares(double dx, double dy)
{
    const auto exponent = [](double d) {
        return static_cast<int>((static_cast<uint32_t>(__double2hiint(d)) >> 20) & 0x7FFu);
    };
    // The high word of the squared significand at 2^62: in [2^60, 2^62). A subnormal difference
    // counts as 2^-1022 at most, whose square is far below kEpsF64.
    const auto square = [](double d) {
        const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d));
        const unsigned long long M = ((b & 0x000FFFFFFFFFFFFFull) | (1ull << 52)) << 10;
        return __umul64hi(M, M);
    };
    const int ex = exponent(dx), ey = exponent(dy), E = max(ex, ey);
    const unsigned long long s =
        (square(dx) >> min(2 * (E - ex), 63)) + (square(dy) >> min(2 * (E - ey), 63));
    const int lz = __clz(static_cast<int>(s >> 32));  // 1 to 3
    const int e = 2 * E - 2043 - lz;
    if (e < -1022)
        return {-1022, 1ull << 63};
    return {e, s << lz};
}

}  // namespace aidw
