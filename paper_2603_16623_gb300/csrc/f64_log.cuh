// f64_log.cuh -- the natural logarithm of the double-precision march.
//
// The table-driven method of P. T. P. Tang, ACM TOMS 16, 1990: x = 2^e m, c
// close to 1/m from a table of 128, ln x = e ln 2 - ln c + log1p(m c - 1).
// c has 8 bits, so that m c - 1 is exact (|m c - 1| < 2^-7), log1p is its
// series (the first term left out is below 2^-59 of it), ln 2 and -ln c come
// in two parts, the high ones multiples of 2^-42 so that e ln 2 - ln c is
// exact in them.  The first interval takes c = 1 and the last two 1/2, whose
// logarithms are exact: around x = 1 nothing is left but the series, and the
// result keeps its full relative accuracy.  What is left are the rounding of
// the sum, 1/2 ulp, and that of the series where -ln c is no larger than it,
// up to 1/4 (measured against 80-bit arithmetic: at most 0.75 ulp, at most
// 0.62 beyond two per cent of 1; the library's log states 1).
// 14 FP64 operations, where the library's log takes a sub-partition's FP64
// pipe for 32 (2050 cycles for a warp).
// The table is computed at compile time, in double-double arithmetic from the
// series -ln c = 2 atanh((1 - c) / (1 + c)).  Compiles for the host too (tests).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define WK_LOG_HD __host__ __device__ __forceinline__
#else
#define WK_LOG_HD inline
#endif

namespace gbwake {

constexpr int kLogCells = 128;
struct F64LogTable {
    double c[kLogCells];                // 1/m to 8 bits
    double h[kLogCells], l[kLogCells];  // -ln c, high (a multiple of 2^-42) and low part
};

namespace f64_log_detail {
struct dd {
    double h, l;
};
constexpr dd quick_sum(double a, double b) {  // |a| >= |b|
    const double s = a + b;
    return {s, b - (s - a)};
}
constexpr dd two_sum(double a, double b) {
    const double s = a + b, t = s - a;
    return {s, (a - (s - t)) + (b - t)};
}
constexpr dd two_prod(double a, double b) {  // (Dekker: the parts have 26 bits)
    const double k = 134217729.0, p = a * b;
    const double ta = k * a, ah = ta - (ta - a), al = a - ah;
    const double tb = k * b, bh = tb - (tb - b), bl = b - bh;
    return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr dd add(dd a, dd b) {
    const dd s = two_sum(a.h, b.h);
    return quick_sum(s.h, s.l + (a.l + b.l));
}
constexpr dd mul(dd a, dd b) {
    const dd p = two_prod(a.h, b.h);
    return quick_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr dd div(dd a, double b) {
    const double q = a.h / b;
    const dd p = two_prod(q, b);
    return quick_sum(q, (((a.h - p.h) - p.l) + a.l) / b);
}
// 2 atanh(a / b) for 0 <= a <= b / 3 (b exact)
constexpr dd two_atanh(double a, double b) {
    const dd s = div({a, 0.0}, b), s2 = mul(s, s);
    dd sum = {0.0, 0.0};
    for (int k = 65; k >= 1; k -= 2) sum = add(mul(sum, s2), div({2.0, 0.0}, (double)k));
    return mul(sum, s);
}
constexpr double kGrid = 6755399441055744.0 / 4398046511104.0;  // 1.5 2^52 / 2^42: adding it rounds to a multiple of 2^-42
constexpr dd split(dd v) {
    const double h = (v.h + kGrid) - kGrid;
    return {h, (v.h - h) + v.l};
}
constexpr dd ln2() { return split(two_atanh(1.0, 3.0)); }
}  // namespace f64_log_detail

constexpr F64LogTable f64_log_table() {
    using namespace f64_log_detail;
    F64LogTable t = {};
    for (int i = 0; i < kLogCells; ++i) {
        dd v = {0.0, 0.0};
        if (i == 0) {
            t.c[i] = 1.0;
        } else if (i >= kLogCells - 2) {
            t.c[i] = 0.5;
            v = ln2();
        } else {
            const int center = 2 * kLogCells + 2 * i + 1;  // the interval's centre x 256
            t.c[i] = (double)((65536 + center / 2) / center) / 256.0;
            v = split(two_atanh(1.0 - t.c[i], 1.0 + t.c[i]));
        }
        t.h[i] = v.h;
        t.l[i] = v.l;
    }
    return t;
}

constexpr double kLn2Hi = f64_log_detail::ln2().h, kLn2Lo = f64_log_detail::ln2().l;

WK_LOG_HD double f64_log(const F64LogTable& t, double x) {
    uint64_t b;
    memcpy(&b, &x, 8);
    const int32_t hi = (int32_t)(b >> 32);
    if ((uint32_t)(hi - 0x00100000) >= 0x7fe00000u) return log(x);  // 0, subnormal, negative, inf, NaN
    const int i = (hi >> 13) & (kLogCells - 1);
    b = (b & 0x000fffffffffffffull) | 0x3ff0000000000000ull;
    double m, e;
    memcpy(&m, &b, 8);
    // the exponent as a double without a conversion: 2^52 + 2^31 + e less 2^52 + 2^31
    b = 0x4330000000000000ull | ((uint32_t)((hi >> 20) - 1023) ^ 0x80000000u);
    memcpy(&e, &b, 8);
    e -= 4503601774854144.0;
    const double z = fma(m, t.c[i], -1.0);
    double p = fma(-0.125, z, 1.0 / 7.0);
    p = fma(p, z, -1.0 / 6.0);
    p = fma(p, z, 0.2);
    p = fma(p, z, -0.25);
    p = fma(p, z, 1.0 / 3.0);
    p = fma(p, z, -0.5);
    const double low = fma(z * z, p, fma(e, kLn2Lo, t.l[i]));
    return fma(e, kLn2Hi, t.h[i]) + (z + low);
}

}  // namespace gbwake
