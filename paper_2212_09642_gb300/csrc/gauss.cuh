// Standard normal probe entries (Box & Muller 1958) with few FP64 operations
// (not part of the public ABI).
//
// x = sqrt(-2 log u1) cos(2 pi u2) in FP64 needs about 80 FP64 instructions with
// the CUDA math library's log, cos and sqrt, and GB300 issues 1.7 FP64 lane
// operations per cycle and SM: 1.25 ms for 9.6 million entries.  Both functions
// are needed on narrow ranges here, so they are taken from tables and short
// series with 33 FP64 instructions and the rest in integer arithmetic,
// accurate to a few units of 2^-53 as before:
//   log u1   u1 = 2^e m, m in [0.75, 1.5); with c_i the reciprocal (to 9 bits) of
//            the middle of m's interval, r = c_i m - 1 (exact to rounding, |r| <
//            2^-7), log u1 = e log 2 - log c_i + log(1 + r) by the power series
//            (table-driven logarithm: P.T.P. Tang, ACM TOMS 16(4), 1990)
//   sqrt     one FP32 reciprocal square root and two corrections
//            s += (y - s s) / (2 s)
//   cos      the angle in 256ths of the circle plus a remainder delta of at most
//            pi / 256: cos(a + d) = cos a + (cos a (cos d - 1) - sin a sin d)
// Tables are built by the compiler from the series below.  Checked on the CPU
// against long double over 2e7 entries: log within 3.1e-16, sqrt within 1.2e-16
// relative, cos within 1.7e-16.  The 9.6 million entries take 0.71 ms.
#pragma once
#include <stdint.h>

namespace vne {

namespace gauss_table {

constexpr double kLn2 = 0.693147180559945309417232121458176568;
constexpr double kTwoPi = 6.28318530717958647692528676655900577;

// log x for x in [0.6, 1.6] by 2 atanh((x - 1) / (x + 1)); long double, so that
// the rounding to double is the only error that matters
constexpr double ct_log(double x) {
    const long double z = ((long double)x - 1.0L) / ((long double)x + 1.0L), z2 = z * z;
    long double t = z, s = 0.0L;
    for (int k = 1; k < 60; k += 2) {
        s += t / k;
        t *= z2;
    }
    return (double)(2.0L * s);
}
constexpr double ct_sin(long double x) {  // |x| <= pi / 4
    long double t = x, s = 0.0L;
    for (int k = 1; k < 40; k += 2) {
        s += t;
        t *= -x * x / ((k + 1) * (k + 2));
    }
    return (double)s;
}
constexpr double ct_cos(long double x) {
    long double t = 1.0L, s = 0.0L;
    for (int k = 0; k < 40; k += 2) {
        s += t;
        t *= -x * x / ((k + 1) * (k + 2));
    }
    return (double)s;
}

struct Tables {
    double log_c[128], log_v[128];  // c_i and -log c_i, i = the top 7 bits of m's fraction
    double cs[256], sn[256];        // cos and sin of 2 pi i / 256
    double ln2e[64];                // -e log 2 for u1 = 2^-e m, e = 0 .. 63
    constexpr Tables() : log_c{}, log_v{}, cs{}, sn{}, ln2e{} {
        for (int i = 0; i < 128; i++) {
            // fraction i / 128 .. (i + 1) / 128 above 1; halves above 1.5
            const double mid = (1.0 + (i + 0.5) / 128.0) * (i >= 64 ? 0.5 : 1.0);
            double c = (double)(int)(512.0 / mid + 0.5) / 512.0;
            if (i == 0 || i == 127) c = 1.0;  // around 1: no table term, so that log 1 = 0 exactly
            log_c[i] = c;
            log_v[i] = c == 1.0 ? 0.0 : -ct_log(c);
        }
        for (int i = 0; i < 256; i++) {
            // octant symmetry keeps the series argument within pi / 4
            const int q = i / 64, k = i % 64;
            const long double pi = 3.14159265358979323846264338327950288L;
            double c = 0.0, s = 0.0;
            if (k <= 32) {
                c = ct_cos(2.0L * pi * k / 256.0L);
                s = ct_sin(2.0L * pi * k / 256.0L);
            } else {
                c = ct_sin(2.0L * pi * (64 - k) / 256.0L);
                s = ct_cos(2.0L * pi * (64 - k) / 256.0L);
            }
            cs[i] = q == 0 ? c : (q == 1 ? -s : (q == 2 ? -c : s));
            sn[i] = q == 0 ? s : (q == 1 ? c : (q == 2 ? -s : -c));
        }
        for (int e = 0; e < 64; e++) ln2e[e] = (double)(-(long double)kLn2 * e);
    }
};

}  // namespace gauss_table

__device__ const gauss_table::Tables kGauss = gauss_table::Tables();

// -log u for u = a double in (0, 1] with exponent >= -63
__device__ __forceinline__ double gauss_neg_log(double u) {
    const uint64_t b = (uint64_t)__double_as_longlong(u);
    const int i = (int)((b >> 45) & 127);
    const int up = i >= 64 ? 1 : 0;                       // m in [1.5, 2) counts as [0.75, 1)
    const int e = 1023 - (int)(b >> 52) - up;             // u = 2^-e m
    const double m = __longlong_as_double((long long)((b & 0x000fffffffffffffULL) | ((uint64_t)(1023 - up) << 52)));
    const double r = fma(m, kGauss.log_c[i], -1.0);
    // log(1 + r) = r - r^2/2 + ... - r^8/8 (|r| < 2^-7: the rest is below 2^-66)
    double p = fma(r, -1.0 / 8.0, 1.0 / 7.0);
    p = fma(r, p, -1.0 / 6.0);
    p = fma(r, p, 1.0 / 5.0);
    p = fma(r, p, -1.0 / 4.0);
    p = fma(r, p, 1.0 / 3.0);
    p = fma(r, p, -0.5);
    p = fma(r * r, p, r);
    return -((kGauss.ln2e[e] + kGauss.log_v[i]) + p);
}

// sqrt y for y in [2^-54, 128), or +-0 (tested by its bits: an FP64 comparison
// would take a slot of the FP64 port)
__device__ __forceinline__ double gauss_sqrt(double y) {
    if ((__double_as_longlong(y) << 1) == 0) return 0.0;
    const float r = rsqrtf((float)y);
    const double h = (double)(0.5f * r);
    double s = y * (double)r;
    s = fma(fma(-s, s, y), h, s);
    return fma(fma(-s, s, y), h, s);
}

// cos(2 pi k / 2^53), k < 2^53
__device__ __forceinline__ double gauss_cos(uint64_t k) {
    const uint64_t kr = k + (1ULL << 44);  // nearest 256th of the circle
    const int i = (int)(kr >> 45) & 255;
    const long long rem = (long long)(kr & ((1ULL << 45) - 1)) - (1LL << 44);
    const double d = (double)rem * (gauss_table::kTwoPi * 0x1.0p-53);
    const double d2 = d * d;
    // cos d - 1 and sin d - d (|d| <= pi / 256: the next terms are below 2^-65)
    const double c1 = d2 * fma(d2, fma(d2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
    const double s3 = d2 * fma(d2, fma(d2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0);
    const double sn = fma(d, s3, d);
    const double C = kGauss.cs[i], S = kGauss.sn[i];
    return fma(-S, sn, fma(C, c1, C));
}

}  // namespace vne
