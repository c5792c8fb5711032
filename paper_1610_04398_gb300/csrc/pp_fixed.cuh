// Fixed-point arithmetic that stands in for FP64 multiply-adds in the long sums of the FP64 path.
// GB300 issues FP64 multiply-adds at 1.67 lanes a clock and SM and 32 x 32 + 64 bit integer ones, two
// instructions each, at 28 (measured), so three integer ones in place of an FP64 one are five times
// faster.  A value is an integer v relative to a common power of two, split v = h 2^28 + l with l in
// [-2^27, 2^27).  Three multiply-adds a product, in 64-bit sums that do not depend on the order:
//   exact (FixedSum):  hh, ll and (h + l)(h' + l') of two values, whose cross terms are the third sum less
//     the other two (Karatsuba and Ofman's product, modulo 2^64: only what is left has to fit);
//   to the cross terms: hh and hl + lh; ll, up to 2^54 of either sign, is dropped: 2^(54 - bits) of a
//     full-scale product of `bits` bits (the translations: 113 bits, 2^-59).
// Rounding the values is then what the sums lose.
#pragma once

#include <cuda_runtime.h>

#include <cstring>

namespace pp {

// s += a b, 32 x 32 + 64 bits, written with the carry (the C expression took about six instructions).
__device__ __forceinline__ void mad_wide(long long& s, int a, int b) {
    int lo = int(s), hi = int(s >> 32);
    asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(b));
    s = (long long)(((unsigned long long)unsigned(hi) << 32) | unsigned(lo));
}

// Halves of v (|v| < 2^58).
__host__ __device__ __forceinline__ int2 split28(long long v) {
    const int l = int(unsigned(v) << 4) >> 4;
    return int2{int((v - l) >> 28), l};
}

// A sum of exact products in units of 2^0: a = sum hh, b = sum ll, c = sum (h + l)(h' + l').
struct FixedSum {
    long long a, b, c;
    __device__ __forceinline__ void clear() { a = b = c = 0; }
    __device__ __forceinline__ void add(int2 q, int qs, int2 k, int ks) {  // qs = q.x + q.y, ks = k.x + k.y
        mad_wide(a, q.x, k.x);
        mad_wide(b, q.y, k.y);
        mad_wide(c, qs, ks);
    }
    // the sum as hi 2^56 + lo 2^28, lo in [0, 2^28) (what is below 2^28 is dropped)
    __device__ __forceinline__ void digits(long long& hi, int& lo) const {
        const long long mid = c - a - b + (b >> 28);
        hi = a + (mid >> 28);
        lo = int(mid) & 0x0fffffff;
    }
};

// Exponent e with |x| < 2^e from the high word of |x|; kExpBad for infinities and NaN, kExpZero for
// zeros and subnormals (they convert to 0).
constexpr int kExpBad = 0x7fffffff, kExpZero = -100000;
__device__ __forceinline__ int exp_of(int hi_abs) {
    return hi_abs >= 0x7ff00000 ? kExpBad : hi_abs < 0x00100000 ? kExpZero : (hi_abs >> 20) - 1022;
}

// x 2^(bits - e) rounded to an integer, for |x| < 2^e and bits <= 57: integer shifts of the
// significand (no FP64 instruction).
__device__ __forceinline__ long long to_fixed(double x, int e, int bits) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
    // x = m 2^(ex - 1075), so x 2^(bits - e) = m 2^-sh, sh >= 53 - bits
    const int sh = e - bits + 1075 - ex;
    if (ex == 0 || sh > 54) return 0;
    const unsigned long long m = (((unsigned long long)(unsigned(hi & 0x000fffff) | 0x00100000u)) << 32) |
                                 (unsigned)__double2loint(x);
    const long long v = (long long)(sh > 0 ? (m + (1ull << (sh - 1))) >> sh : m << -sh);
    return hi < 0 ? -v : v;
}

// 2^e as a double, e in [-1022, 1023] (clamped).
__host__ __device__ __forceinline__ double pow2(int e) {
    e = e < -1022 ? -1022 : e > 1023 ? 1023 : e;
    const unsigned long long b = (unsigned long long)(e + 1023) << 52;
    double d;
    memcpy(&d, &b, 8);
    return d;
}

}  // namespace pp
