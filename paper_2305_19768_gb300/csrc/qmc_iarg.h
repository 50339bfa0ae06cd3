// Argument of x + i y on the integer pipe, for sums of arguments whose small
// values count: relative error below 2^-55 whatever the size, added up in
// 128-bit fixed point (2^-120, so that a sum has FP64's precision down to 2^-66).
//
// With mn <= mx the smaller and larger of |x|, |y| and c = j/64 nearest mn/mx
// (j from an FP32 estimate), atan(mn/mx) = atan(c) + atan(d),
// d = (mn - c mx) / (mx + c mn), |d| <= 2^-7, and atan(d) = d - d^3 (1/3 -
// d^2 (1/5 - d^2 / 7)) (truncation below 2^-66 relative), the inner
// coefficients in 32 bits. For j > 0 the result is at least 2^-7 and is summed
// in Q63; for j = 0 it is d itself, kept as mantissa and exponent. Then the
// octant: pi/2 - r where |y| > |x|, pi - r where x < 0, and the sign of y.
//
// Written for both the device and a host compiler.
#pragma once
#include "qmc_xf.h"

#define QMC_IARG_PI2_61 0x3243F6A8885A308DULL   // RN(2^61 pi / 2)
#define QMC_IARG_PI_61 0x6487ED5110B4611AULL    // RN(2^61 pi)

// tab: RN(2^63 atan(j / 64)), j = 0..64. In (-pi, pi]; with m0 a zero y counts
// as -0 (the prescription F - i0). (0, 0) gives 0. The mantissa is not normalised.
QMC_HD qmc_xf qmc_iarg(double y, double x, bool m0, const int64_t *tab) {
    const qmc_xf ax = qmc_xf_of(x), ay = qmc_xf_of(y);
    const bool sw = ay.e > ax.e || (ay.e == ax.e && ay.m > ax.m);
    const uint64_t mx = sw ? ay.m : ax.m, ms = sw ? ax.m : ay.m;
    const int dd = sw ? ay.e - ax.e : ax.e - ay.e;
    uint64_t dm = 0;                                   // the result, dm 2^(de - 63)
    int de = 0;
    if (mx != 0 && ms != 0) {
        int j = 0;
        if (dd <= 7) {
            // 64 mn / mx within 2^-20
#if defined(__CUDA_ARCH__)
            const float fs = __int_as_float(0x3F800000 | (int)((ms >> 40) & 0x7FFFFFu));
            const float fx = __int_as_float(0x3F800000 | (int)((mx >> 40) & 0x7FFFFFu));
            j = min(__float2int_rn(__fdividef(fs, fx) * __int_as_float((133 - dd) << 23)), 64);
#else
            j = (int)((float)(ms >> 40) / (float)(mx >> 40) * (64 >> dd > 0 ? (float)(64 >> dd) : 0.5f) + 0.5f);
            if (j > 64) j = 64;
#endif
        }
        // one reciprocal and one product for both cases; for j > 0 in units of
        // mx's last place, halved so that the difference (up to mx / 2) keeps its sign
        const uint64_t mn = j ? ms >> dd : 0;
        const int64_t num = (int64_t)((mn >> 1 << 6) - (uint64_t)j * (mx >> 1));       // 32 (mn - c mx)
        const bool below = num < 0;                                                    // d < 0
        const uint64_t den = (mx >> 1) + qmc_umulhi64(mn, (uint64_t)j << 57);          // (mx + c mn) / 2
        const int c = qmc_clz64(den);
        const qmc_xf q = qmc_xf_rcp3(qmc_xf{den << c, 0, 0});                          // 2^63 / (den 2^c)
        const uint64_t p = qmc_umulhi64(j ? (uint64_t)(below ? -num : num) : ms, q.m);
        // |d|: dm 2^-70 for j > 0, else dm 2^(de - 63) with dm normalised; D = |d| 2^70
        const int top = (int)(p >> 63);
        de = q.e + top - dd;                                                           // j = 0: <= -7
        dm = p << (j ? q.e + 2 + c : 1 - top);
        const uint64_t D = j ? dm : (de > -71 ? dm >> (-7 - de) : 0);
        // atan(d) = d (1 - k), k in Q64
        const uint64_t z = qmc_umulhi64(D, D);         // d^2 2^76
        const uint32_t z45 = (uint32_t)(z >> 31);
        const uint32_t c5 = 0x33333333u - (qmc_umulhi32(z45, 0x24924925u) >> 13);
        const uint64_t c3 = 0x2AAAAAAAAAAAAAABULL - (((uint64_t)z45 * c5) >> 14);
        dm -= qmc_umulhi64(dm, qmc_umulhi64(z, c3) >> 11);
        if (j) {
            dm = (uint64_t)tab[j] + (below ? 0 - (dm >> 7) : dm >> 7);
            de = 0;
        }
    }
    if (sw || ax.neg) {
        uint64_t v = de > -62 ? dm >> (2 - de) : 0;    // Q61
        if (sw) v = QMC_IARG_PI2_61 - v;
        if (ax.neg) v = QMC_IARG_PI_61 - v;
        dm = v;
        de = 2;
    }
    return qmc_xf{dm, de, (ay.neg || (m0 && ay.m == 0)) ? 1 : 0};
}

// sum + k a for such an argument a, |k| <= 4, sum in units of 2^-120 modulo 2^128
QMC_HD qmc_u128 qmc_iarg_add(qmc_u128 sum, qmc_xf a, int k) {
    qmc_u128 v = 0;
    if (a.e >= -57) v = (qmc_u128)a.m << (57 + a.e);
    else if (a.e > -121) v = a.m >> (-57 - a.e);
    const int n = a.neg ? -k : k;
    return n < 0 ? sum - v * (uint32_t)-n : sum + v * (uint32_t)n;
}

// RN of a sum
QMC_HD double qmc_iarg_sum(qmc_u128 sum) {
    const bool neg = (sum >> 127) != 0;
    if (neg) sum = 0 - sum;
    const uint64_t hi = (uint64_t)(sum >> 64);
    const int c = hi ? qmc_clz64(hi) : 64 + qmc_clz64((uint64_t)sum);
    if (c == 128) return 0.0;
    sum <<= c;
    return qmc_xf_to_double(qmc_xf{(uint64_t)(sum >> 64) | ((uint64_t)sum ? 1 : 0), 7 - c, neg ? 1 : 0});
}
