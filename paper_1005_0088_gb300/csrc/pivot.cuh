// Arithmetic of the pivots of the diagonal blocks (device code).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace ndsi {

// |p|^2 of a pivot that cannot be inverted: zero or non-finite (decided on its bits, off the FP64 pipe).
__device__ __forceinline__ bool bad_pivot(double den) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(den)) & 0x7FFFFFFFu;
    return hi >= 0x7FF00000u || (hi | static_cast<uint32_t>(__double2loint(den))) == 0;
}

// 1 / x for x > 0, correctly rounded but for results within 2^-9 units in the last place of a tie (outside the
// normal range by division): the hardware's FP32 reciprocal of the mantissa (relative error e below 2^-21) and
// one third-order step y (1 + e + e^2), e = 1 - m y (the series of 1 / (1 - e); what is left is e^3 < 2^-63).  A
// division takes 435 clocks, FP64 instructions of one warp 64 each.
__device__ __forceinline__ double pivot_rcp(double x) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
    const uint32_t ex = hi >> 20;
    if (ex - 1u >= 2044u) return 1.0 / x;  // zero, subnormal, non-finite, or a subnormal result
    const double m = __hiloint2double(static_cast<int>((hi & 0xFFFFFu) | 0x3FF00000u), static_cast<int>(lo));
    const float mf = __uint_as_float(0x3F800000u | (hi & 0xFFFFFu) << 3 | lo >> 29);
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(mf));
    const uint32_t yb = __float_as_uint(yf);
    const double y = __hiloint2double(static_cast<int>((yb >> 3) + (896u << 20)), static_cast<int>(yb << 29));
    const double e = fma(-m, y, 1.0);
    const double r = fma(y, fma(e, e, e), y);  // in [1/2, 1]
    return __hiloint2double(__double2hiint(r) - ((static_cast<int>(ex) - 1023) << 20), __double2loint(r));
}

}  // namespace ndsi
