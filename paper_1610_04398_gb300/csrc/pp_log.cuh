// Natural logarithm in FP64 from a table, for sums of q log r on GB300's narrow FP64 pipe (an
// FP64 instruction occupies an SM's pipe for about 19 cycles, so the library's log, some thirty
// of them, is what the direct sums and multipole evaluations spend their time on).  Table-driven
// method of Tang (ACM TOMS 16, 1990): x = 2^e m, m in [1, 2), c the reciprocal of the midpoint of m's
// 1/256 bin to ten bits, 1 in the first bin and 1/2 in the last, r = m c - 1 (one fused multiply-add, at
// most 2^-8), and with e + 1 and 2 c in place of e and c where m is above 1 + 106/256 (about sqrt 2)
//   log x = e log 2 - log c + (r - r^2/2 + ... + r^7/7)   (truncation below 2^-67):
// ten FP64 instructions.  c is exact and |log c| at most 0.35, so the result keeps its relative accuracy
// around 1: within 1.4 units in the last place.
// Subnormal, infinite, NaN and non-positive arguments take the library's log.
#pragma once

#include <cuda_runtime.h>

namespace pp {

struct LogTable {
    static constexpr int kSplit = 106;  // bins from here on: e + 1
    double c[256], lc[256];  // c, -log c or -log 2c
    constexpr LogTable() : c(), lc() {
        for (int i = 0; i < 256; ++i) {
            const double x = (i + 0.5) / 256.0;
            const int k = int(1024.0 / (1.0 + x) + 0.5);
            c[i] = i == 0 ? 1.0 : i == 255 ? 0.5 : k / 1024.0;
            // -log d = 2 atanh z, z = (1 - d) / (1 + d) = z + dz (the quotient's remainder is exact in two
            // halves of z), |z| < 0.18: z first, the rest of the series is at most 1% of it
            const double d = i < kSplit ? c[i] : 2.0 * c[i], a = 1.0 - d, b = 1.0 + d, z = a / b;
            const double zh = double(int(z * 67108864.0)) / 67108864.0, zl = z - zh;
            const double dz = (a - zh * b - zl * b) / b, z2 = z * z;
            double s = 0.0;
            for (int n = 16; n >= 1; --n) s = (s + 1.0 / (2 * n + 1)) * z2;
            lc[i] = 2.0 * (z + (dz + z * s));
        }
    }
};
static __device__ const LogTable g_log_table = LogTable();

__device__ __forceinline__ double log_table(double x) {
    const int hi = __double2hiint(x);
    if (unsigned(hi) - 0x00100000u >= 0x7fe00000u) return log(x);
    const int i = (hi >> 12) & 255;
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    // e + 2^52 + 2^31 as a double, then e (one addition in place of a conversion)
    const int ei = ((hi + ((256 - LogTable::kSplit) << 12)) >> 20) - 1023;
    const double e = __hiloint2double(0x43300000, ei ^ 0x80000000) - 4503601774854144.0;
    const double r = fma(m, __ldg(&g_log_table.c[i]), -1.0);
    double s = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    s = fma(r, s, 0.2);
    s = fma(r, s, -0.25);
    s = fma(r, s, 1.0 / 3.0);
    s = fma(r, s, -0.5);
    s = fma(r * r, s, r);
    // the small terms first: one rounding at the size of the result
    return fma(e, 0.69314718055994530941723212145818, __ldg(&g_log_table.lc[i]) + s);
}

}  // namespace pp
