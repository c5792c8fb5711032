// Natural logarithm in FP64 from a table, for sums of q log r on GB300's narrow FP64 pipe (an
// FP64 instruction occupies an SM's pipe for about 19 cycles, so the library's log, some thirty
// of them, is what the direct sums and multipole evaluations spend their time on).  Table-driven
// method of Tang (ACM TOMS 16, 1990): x = 2^e m, m in [1, 2), F the midpoint of m's 1/128 bin,
// c = 1 / F rounded, r = m c - 1 (one fused multiply-add, |r| < 2^-8), and
//   log x = e log 2 + log F + (r - r^2/2 + ... + r^7/7)   (truncation below 2^-66):
// ten FP64 instructions.  The absolute error is that of rounding the result (about one unit in
// the last place of max(|log x|, 0.7)), which is what a sum of many logarithms sees.
// Subnormal, infinite, NaN and non-positive arguments take the library's log.
#pragma once

#include <cuda_runtime.h>

namespace pp {

struct LogTable {
    double c[128], lf[128];
    constexpr LogTable() : c(), lf() {
        for (int i = 0; i < 128; ++i) {
            const double x = (i + 0.5) / 128.0, z = x / (2.0 + x), z2 = z * z;
            c[i] = 1.0 / (1.0 + x);
            double s = 0.0;  // log(1 + x) = 2 atanh z = 2 z sum z^2n / (2n + 1), z <= 1/3
            for (int n = 20; n >= 0; --n) s = s * z2 + 1.0 / (2 * n + 1);
            lf[i] = 2.0 * z * s;
        }
    }
};
static __device__ const LogTable g_log_table = LogTable();

__device__ __forceinline__ double log_table(double x) {
    const int hi = __double2hiint(x);
    if (unsigned(hi) - 0x00100000u >= 0x7fe00000u) return log(x);
    const int i = (hi >> 13) & 127;
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    // e + 2^52 + 2^31 as a double, then e (one addition in place of a conversion)
    const double e = __hiloint2double(0x43300000, ((hi >> 20) - 1023) ^ 0x80000000) - 4503601774854144.0;
    const double r = fma(m, __ldg(&g_log_table.c[i]), -1.0);
    double s = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    s = fma(r, s, 0.2);
    s = fma(r, s, -0.25);
    s = fma(r, s, 1.0 / 3.0);
    s = fma(r, s, -0.5);
    s = fma(r * r, s, r);
    return fma(e, 0.69314718055994530941723212145818, __ldg(&g_log_table.lf[i])) + s;
}

}  // namespace pp
