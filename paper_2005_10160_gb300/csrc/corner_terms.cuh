// FP64 logarithm and arc tangent for the prism corner terms (Eq. 2), with few
// FP64 instructions: on this GPU they run at 1/64 of the FP32 rate, and the
// corner terms are all that bounds kernel generation.
//
// Both use a table and a short Taylor series (table-driven evaluation in the
// manner of P. T. P. Tang, ACM TOMS 16 (1990) 378-400 and 18 (1992) 211-222):
//   log1p(u) for u >= 0: w = 1 + u = 2^k m, m in [1, 2); with c close to 1 / m
//     of few bits (c = 1 in the first interval),
//     log w = k ln 2 - log c + log1p(m c - 1 + (what 1 + u rounded off) c / 2^k),
//     the last by the Mercator series of degree 8 (its argument is below
//     2^-7).  In the first interval the first two terms are 0, so small u keep
//     their relative accuracy.
//   atan(a / b) for a, b > 0: t = min / max is close to j / 64, and
//     atan t = atan(j / 64) + atan((min - max j / 64) / (max + min j / 64)), the
//     last by the Gregory series of degree 9 (argument below 1 / 128); for
//     a > b, pi / 2 minus that.  j = 0 keeps the relative accuracy of small t.
// The tables are built once per CTA with the library functions log and atan.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace grav {

struct CornerTables {
    static constexpr int LOGS = 128, ATANS = 65;
    double c[LOGS], mlogc[LOGS];  // c and -log c per interval of m
    double at[ATANS];             // atan(j / 64)
};

// Entry e of the tables.
__host__ __device__ inline void corner_table_entry(CornerTables& t, int e) {
    if (e < CornerTables::LOGS) {
        // 1 / (midpoint), rounded to 10 bits so that m c - 1 loses nothing
        const double mid = 1.0 + (e + 0.5) / CornerTables::LOGS;
        const double c = e == 0 ? 1.0 : floor(1024.0 / mid + 0.5) / 1024.0;
        t.c[e] = c;
        t.mlogc[e] = e == 0 ? 0.0 : -log(c);
    }
    if (e < CornerTables::ATANS) t.at[e] = atan(e / 64.0);
}

__host__ __device__ __forceinline__ uint64_t bits_of(double v) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t b;
    memcpy(&b, &v, 8);
    return b;
#endif
}
__host__ __device__ __forceinline__ double of_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    memcpy(&v, &b, 8);
    return v;
#endif
}

// log(1 + u), u >= 0 and finite.
__host__ __device__ __forceinline__ double log1p_pos(double u, const CornerTables& t) {
    const double w = 1.0 + u;
    const double lost = u < 1.0 ? u - (w - 1.0) : 1.0 - (w - u);  // 1 + u = w + lost exactly
    const uint64_t wb = bits_of(w);
    const int k = (int)(wb >> 52) - 1023;
    const int i = (int)(wb >> 45) & 127;
    const double m = of_bits((wb & 0xfffffffffffffull) | 0x3ff0000000000000ull);
    const double scale = of_bits((uint64_t)(1023 - k) << 52);  // 2^-k, k < 1023
    const double c = t.c[i];
    const double r = fma(lost * scale, c, fma(m, c, -1.0));
    double p = -1.0 / 8.0;
    p = fma(p, r, 1.0 / 7.0);
    p = fma(p, r, -1.0 / 6.0);
    p = fma(p, r, 1.0 / 5.0);
    p = fma(p, r, -1.0 / 4.0);
    p = fma(p, r, 1.0 / 3.0);
    p = fma(p, r, -1.0 / 2.0);
    const double tail = fma(p, r * r, r);
    return fma((double)k, 0.69314718055994530942, t.mlogc[i]) + tail;
}

// a / b to a few bits for 0 < a <= b, by integer arithmetic on the exponents
// (no FP64 instruction, and no range lost to FP32).
__host__ __device__ __forceinline__ float coarse_ratio(double a, double b) {
    const uint64_t ab = bits_of(a), bb = bits_of(b);
    const int de = (int)(ab >> 52) - (int)(bb >> 52);  // <= 0
    if (de < -12) return 0.f;
    const uint32_t am = 0x3f800000u | (uint32_t)((ab >> 29) & 0x7fffffu), bm = 0x3f800000u | (uint32_t)((bb >> 29) & 0x7fffffu);
    float fa, fb;
#ifdef __CUDA_ARCH__
    fa = __uint_as_float(am + ((uint32_t)de << 23));
    fb = __uint_as_float(bm);
    return __fdividef(fa, fb);
#else
    const uint32_t as = am + ((uint32_t)de << 23);
    memcpy(&fa, &as, 4);
    memcpy(&fb, &bm, 4);
    return fa / fb;
#endif
}

// atan(a / b), a, b > 0 and finite.
__host__ __device__ __forceinline__ double atan_ratio(double a, double b, const CornerTables& t) {
    const bool swap = a > b;
    const double lo = swap ? b : a, hi = swap ? a : b;
    const int j = (int)(coarse_ratio(lo, hi) * 64.f + 0.5f);  // 0 .. 64
    const double c = (double)((float)j * 0.015625f);
    const double s = fma(-c, hi, lo) / fma(c, lo, hi);
    const double z = s * s;
    double p = 1.0 / 9.0;
    p = fma(p, z, -1.0 / 7.0);
    p = fma(p, z, 1.0 / 5.0);
    p = fma(p, z, -1.0 / 3.0);
    const double v = t.at[j] + fma(p * z, s, s);
    return swap ? 1.57079632679489661923 - v : v;
}

}  // namespace grav
