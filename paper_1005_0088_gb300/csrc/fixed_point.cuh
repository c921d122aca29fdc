// Exact fixed-point sums of complex products on the integer multiply-add pipe (device code).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace ndsi {

// Fixed-point products.  GB300 issues one warp-wide FP64 instruction per SM every 16-19 clocks (1.7-2
// lanes a clock; 64 clocks per sub-partition) but 59 lanes a clock of 32 x 32 + 64-bit integer
// multiply-adds (both measured), so products of complex matrices are formed in fixed point: over a
// chunk of inner indices every row of op(A) and column of op(B) is scaled by a power of two and cut to
// two integer digits, x = (h 2^LB + l) 2^(E - 2 LB + 1), and integer multiply-adds sum h h and h l + l h
// exactly in 64 bits; l l is dropped, and the sum is rounded once to FP64.  Two forms:
//  * the GEMMs and the diagonal blocks: LB = 28 (55 bits), chunks of at most 64 indices, three real
//    products per complex one (Fix3Sum, below);
//  * the solves: LB = 29 (57 bits), chunks of 16, four real products (FixSum): |h| <= 2^28 and
//    -2^28 <= l < 2^28, so that over kFixK = 32 terms the sums stay within 2^62 (h h) and 2^63.
// The error of an output is about 2^-(2 LB - 1) of (row maximum) x (column maximum) per term and one
// rounding per chunk, against one FP64 rounding of every term in a DFMA loop: the bits of elements far below
// their row's maximum are lost.  The basis functions are therefore brought to a common scale beforehand
// (launch_basis_scale), so that a row's maximum speaks for the row; elements below 2^-(2 LB - 1) of it and
// subnormal ones count as zero.  Rows or columns holding an infinity or NaN give NaN.
constexpr int kFixK = 32;          // inner indices the four-product sums (FixSum) are exact over
constexpr int kFixNonFinite = 1 << 20;  // row exponent of a row holding an infinity or NaN

// Digits of x at row exponent field `emax` (x == 0 or its exponent field <= emax), LB bits in the low one:
// F = x 2^(2 LB - 1 - E) cut towards zero = h 2^LB + l.
template <int LB = 29>
__device__ __forceinline__ void fix_digits(double x, int emax, int& h, int& l) {
    const int64_t b = __double_as_longlong(x);
    const int ex = static_cast<int>((b >> 52) & 0x7FF);
    const uint64_t m = (static_cast<uint64_t>(b) << 10 & 0x3FFFFFFFFFFFFFFFull) | 0x4000000000000000ull;  // 1.f at bit 62
    const int sh = ex ? min(64 - 2 * LB + emax - ex, 63) : 63;
    int64_t f = static_cast<int64_t>(m >> sh);
    f = b < 0 ? -f : f;
    l = static_cast<int>(static_cast<uint32_t>(f) << (32 - LB)) >> (32 - LB);
    h = static_cast<int>((f - l) >> LB);
    // plain 32-bit values from here on: products of digits still in registers stay single wide
    // multiply-adds instead of 64-bit multiplications
    asm("" : "+r"(h), "+r"(l));
}

template <int LB>
static __device__ __noinline__ double fix_to_double_slow(int64_t t, uint32_t rem, int e) {
    if (e >= kFixNonFinite / 2) return __longlong_as_double(0x7FF8000000000000ll);
    return ldexp(ldexp(static_cast<double>(t), LB) + static_cast<double>(rem), e + LB);
}
// (hh 2^(2 LB) + mid 2^LB) 2^e rounded to FP64, with integer operations.
template <int LB = 29>
__device__ __forceinline__ double fix_to_double(int64_t hh, int64_t mid, int e) {
    constexpr uint32_t mask = (1u << LB) - 1;
    const int64_t t = hh + (mid >> LB);
    const uint32_t rem = static_cast<uint32_t>(mid) & mask;
    const bool neg = t < 0;
    const uint64_t tm = static_cast<uint64_t>(neg ? (rem ? ~t : -t) : t);
    const uint32_t rm = neg ? (mask + 1 - rem) & mask : rem;
    const int s = min(__clzll(static_cast<long long>(tm)), LB);
    uint64_t u = (tm << s) | (rm >> (LB - s));
    const int lz = __clzll(static_cast<long long>(u));
    const int biased = 63 - lz + 2 * LB - s + e + 1023;
    if (biased <= 0 || biased >= 2046) return u || e >= kFixNonFinite / 2 ? fix_to_double_slow<LB>(t, rem, e) : 0.0;
    u <<= lz & 63;
    const uint64_t mant = (u >> 11) + ((u >> 10) & 1);  // in [2^52, 2^53]; zero when u is
    const uint64_t bits = u ? (static_cast<uint64_t>(biased - 1) << 52) + mant : 0;
    return __longlong_as_double(static_cast<int64_t>(bits | static_cast<uint64_t>(neg) << 63));
}

// One complex product into the four exact sums: (a.x + i a.z) (b.x + i b.z) with low digits y, w.
struct FixSum {
    int64_t rh, rm, ih, im;
};
__device__ __forceinline__ void fix_mac(FixSum& c, const int4& a, const int4& b) {
    const int nzh = -a.z, nzl = -a.w;
    c.rh += static_cast<int64_t>(a.x) * b.x;
    c.rm += static_cast<int64_t>(a.x) * b.y;
    c.ih += static_cast<int64_t>(a.x) * b.z;
    c.im += static_cast<int64_t>(a.x) * b.w;
    c.rm += static_cast<int64_t>(a.y) * b.x;
    c.im += static_cast<int64_t>(a.y) * b.z;
    c.ih += static_cast<int64_t>(a.z) * b.x;
    c.im += static_cast<int64_t>(a.z) * b.y;
    c.rh += static_cast<int64_t>(nzh) * b.z;
    c.rm += static_cast<int64_t>(nzh) * b.w;
    c.im += static_cast<int64_t>(a.w) * b.x;
    c.rm += static_cast<int64_t>(nzl) * b.z;
}
__device__ __forceinline__ double2 fix_value(const FixSum& c, int e) {
    return make_double2(fix_to_double(c.rh, c.rm, e), fix_to_double(c.ih, c.im, e));
}
__device__ __forceinline__ int expo_bits(double2 v) {
    return max(__double2hiint(v.x) & 0x7FF00000, __double2hiint(v.y) & 0x7FF00000);
}
template <int LB = 29>
__device__ __forceinline__ int4 fix_digits2(double2 v, int emax) {
    int4 q;
    fix_digits<LB>(v.x, emax, q.x, q.y);
    fix_digits<LB>(v.y, emax, q.z, q.w);
    return q;
}
// Exponent a row's digits are stored with, from its largest exponent field.
template <int LB = 29>
__device__ __forceinline__ int fix_expo(int emax) {
    return emax == 0x7FF ? kFixNonFinite : emax - 1022 - (2 * LB - 1);
}

// The same with three real products per complex one (Re = P1 - P2, Im = P3 - P1 - P2, P3 = (Ar + Ai)(Br + Bi)):
// nine multiply-adds instead of twelve.  28-bit low digits (55 bits in all) keep the sums of two digits
// in 32 bits; the sums count modulo 2^64, and the differences that are wanted lie within 2 2^54 (h h)
// and 4 2^54 (h l + l h) per term, so that they are exact over kFix3K terms (2^61 and 2^62).
// Dropping l l and the cut at 2^-55 of the row maximum leave the errors of whole sweeps as they were
// (7.2e-15 for a 32 x 32 x 4 sheet, 1.3e-14 for Green functions of a 9 x 8 x 7 x 5 box; DFMA loops
// 7.2e-15 and 1.4e-14): the FP64 sums around the products decide them.
constexpr int kFix3 = 28;
constexpr int kFix3K = 64;
struct Fix3Sum {
    uint64_t h1, m1, h2, m2, h3, m3;
};
__device__ __forceinline__ uint64_t fix_wide(int a, int b) { return static_cast<uint64_t>(static_cast<int64_t>(a) * b); }
__device__ __forceinline__ void fix3_mac(Fix3Sum& c, const int4& a, int2 as, const int4& b, int2 bs) {
    c.h1 += fix_wide(a.x, b.x);
    c.m1 += fix_wide(a.x, b.y);
    c.m1 += fix_wide(a.y, b.x);
    c.h2 += fix_wide(a.z, b.z);
    c.m2 += fix_wide(a.z, b.w);
    c.m2 += fix_wide(a.w, b.z);
    c.h3 += fix_wide(as.x, bs.x);
    c.m3 += fix_wide(as.x, bs.y);
    c.m3 += fix_wide(as.y, bs.x);
}
__device__ __forceinline__ int2 fix3_sum(const int4& a) { return make_int2(a.x + a.z, a.y + a.w); }
__device__ __forceinline__ void fix3_mac(Fix3Sum& c, const int4& a, const int4& b) {
    fix3_mac(c, a, fix3_sum(a), b, fix3_sum(b));
}
__device__ __forceinline__ double2 fix3_value(const Fix3Sum& c, int e) {
    return make_double2(fix_to_double<kFix3>(static_cast<int64_t>(c.h1 - c.h2), static_cast<int64_t>(c.m1 - c.m2), e),
                        fix_to_double<kFix3>(static_cast<int64_t>(c.h3 - c.h1 - c.h2),
                                             static_cast<int64_t>(c.m3 - c.m1 - c.m2), e));
}

}  // namespace ndsi
