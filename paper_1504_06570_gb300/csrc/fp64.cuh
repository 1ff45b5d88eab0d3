// FP64 helpers of the photon path for a GPU whose FP64 pipe is its bottleneck.
//
// On GB300 a warp's FP64 instruction holds the SM's FP64 pipe for sixteen cycles (1.06 TFLOP/s measured, against
// 77 for FP32), and a conversion to or from double or a double comparison costs as much as a fused
// multiply-add; the FP64 kernels keep that pipe 86 % busy while the integer and FP32 pipes idle.  So reciprocals
// and roots start from the hardware's approximations (PTX rcp.approx.ftz.f64 and rsqrt.approx.ftz.f64, about 20
// bits, not on the FP64 pipe) and take one step of third order (Householder's iteration), which leaves a
// relative error near 2^-60 before rounding, and conversions are integer operations on the words of a double.
// Arguments are finite, non-zero and far from the ends of the exponent range where not said otherwise.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

namespace phosim {

// 1 / b: with r = 1 - b x the exact reciprocal is x / (1 - r) = x (1 + r + r^2 + ...)
__device__ __forceinline__ double rcp64(double b) {
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(b));
    const double r = fma(-b, x, 1.0);
    return fma(x, fma(r, r, r), x);
}

__device__ __forceinline__ double rsqrt_seed64(double a) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    return y;
}
// 1 / sqrt(a), a > 0: with e = 1 - a y^2 it is y (1 - e)^(-1/2) = y (1 + e / 2 + 3 e^2 / 8 + ...)
__device__ __forceinline__ double rsqrt64(double a) {
    const double y = rsqrt_seed64(a), e = fma(-(a * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
// sqrt(a), a > 0, from s = a y the same way
__device__ __forceinline__ double sqrt64_pos(double a) {
    const double y = rsqrt_seed64(a), s = a * y, e = fma(-s, y, 1.0);
    return fma(s * e, fma(0.375, e, 0.5), s);
}
// sign tests on the high word, and 0 <= a < b for b > 0 by the order of the words (a double comparison takes the FP64
// pipe); -0 is 0, and a NaN is not below
__device__ __forceinline__ bool negative64(double a) { return __double2hiint(a) < 0; }
__device__ __forceinline__ bool within64(double a, double b) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(a);
    return u < (unsigned long long)__double_as_longlong(b) || u == 1ull << 63;
}
// sqrt(a) for a >= 0; numbers below 1e-290 give 0
__device__ __forceinline__ double sqrt64(double a) { return __double2hiint(a) > 0x03c00000 ? sqrt64_pos(a) : 0.0; }

// a double truncated to single precision; magnitudes below 1e-38 give a number of that size, those above 3e38 the
// largest float (a start value or a comparison with a margin, never a result)
__device__ __forceinline__ float f32_trunc(double v) {
    const int hi = __double2hiint(v);
    int m = hi & 0x7fffffff;
    m = m < 0x38000000 ? 0x38000000 : (m > 0x47efffff ? 0x47efffff : m);
    const uint32_t bits = __funnelshift_l((uint32_t)__double2loint(v), (uint32_t)(m - 0x38000000), 3);
    return __uint_as_float((bits & 0x7fffffffu) | ((uint32_t)hi & 0x80000000u));
}
// (float)v, rounded to nearest even, for 0 or 1e-37 < v (infinity above 3.4e38)
__device__ __forceinline__ float f32_rn_pos(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    if (hi < 0x38100000u) return 0.f;
    if (hi >= 0x47f00000u) return INFINITY;
    const unsigned long long b = ((unsigned long long)(hi - 0x38000000u) << 32) | lo;
    return __uint_as_float((uint32_t)((b + 0x0fffffffull + ((lo >> 29) & 1u)) >> 29));
}
// (double)f, exact, for 0 and normal finite numbers
__device__ __forceinline__ double f64_exact(float f) {
    const uint32_t b = __float_as_uint(f), m = b & 0x7fffffffu;
    const uint32_t hi = m ? (b & 0x80000000u) | ((m >> 3) + 0x38000000u) : b;
    return __hiloint2double((int)hi, (int)(b << 29));
}
// the same for any normal number, infinity or NaN
__device__ __forceinline__ double f64_any(float f) {
    const uint32_t b = __float_as_uint(f), m = b & 0x7fffffffu;
    uint32_t hi = m ? (b & 0x80000000u) | ((m >> 3) + 0x38000000u) : b;
    if (m >= 0x7f800000u) hi |= 0x7ff00000u;
    return __hiloint2double((int)hi, (int)(b << 29));
}
// (double)n of a non-negative n, exact: 2^52 + n by its bits, then 2^52 off
__device__ __forceinline__ double f64_of_count(uint32_t n) { return __hiloint2double(0x43300000, (int)n) - 4503599627370496.0; }

// floor(s k) as a double and an integer: the product added to 1.5 2^52 and rounded down in one operation leaves the
// integer in the low word.  False where the floor is not a signed 32-bit integer (nothing is set then): the high word
// holds all that is above the low one, so it is 0x43380000 less the low word's sign.
__device__ __forceinline__ bool floor_product64(double s, double k, double& fl, int& i) {
    const double t = __fma_rd(s, k, 6755399441055744.0);
    const int low = __double2loint(t);
    if (__double2hiint(t) != 0x43380000 + (low >> 31)) return false;
    fl = t - 6755399441055744.0;
    i = low;
    return true;
}

// s k for a factor k = m 2^(E - 63) (m its significand in the top 53 bits, factor64) by integers: the floor, and the first
// 52 bits after it.  s is taken to 2^-40 (finer than the rounding of a position in millimetres beyond 4 m) and below 2^22;
// false beyond, or where the factor has no integer form (shift 0).
__device__ __forceinline__ bool split_product64(double s, unsigned long long m, int shift, int& i, unsigned long long& frac) {
    const uint32_t hi = (uint32_t)__double2hiint(s), lo = (uint32_t)__double2loint(s), e = (hi >> 20) & 0x7ffu;
    if (e >= 1023u + 22u || shift == 0) return false;
    // |s| = norm 2^(e - 1023 - 63), and in units of 2^-40
    const unsigned long long norm = ((unsigned long long)(((hi & 0xfffffu) | 0x100000u) << 11 | lo >> 21) << 32) | (unsigned long long)(lo << 11);
    const unsigned long long fixed = norm >> min(1023u + 23u - e, 63u);
    unsigned long long ph = __umul64hi(fixed, m), pl = fixed * m;
    if ((int)hi < 0) { pl = 0ull - pl; ph = ~ph + (pl == 0ull); }
    i = (int)((long long)ph >> (shift - 12));
    frac = shift < 64 ? (ph << (64 - shift)) | (pl >> shift) : (unsigned long long)((long long)ph >> (shift - 64));
    frac &= 0xfffffffffffffull;
    return true;
}
// 1 + the fraction of 52 bits, exact; kNoFraction gives a NaN, here and in single precision
constexpr unsigned long long kNoFraction = ~0ull;
__device__ __forceinline__ double one_and_fraction64(unsigned long long frac) {
    return __longlong_as_double((long long)(frac | 0x3ff0000000000000ull));
}
// the fraction in single precision, rounded to nearest (above 2^-21): its first 23 bits, and the next 23 with a last one
// that says whether any is left, which are exact, in one sum
__device__ __forceinline__ float fraction_f32(unsigned long long frac) {
    const uint32_t head = (uint32_t)(frac >> 29), tail = (uint32_t)frac & 0x1fffffffu;
    const float f = fmaf((float)(tail >> 5 | (uint32_t)((tail & 31u) != 0u)), 0x1p-47f, (float)head * 0x1p-23f);
    return head >> 23 ? __uint_as_float(0x7fffffffu) : f;
}
// log((w + 1/2) 2^-32) by a table (Tang 1990): with (w + 1/2) 2^-32 = 2^-e m, m in [1, 2), c near 1 / m from the first 8
// bits after m's leading one and r = m c - 1, exact, it is -e log 2 - log c + log(1 + r); from m = sqrt 2 on the table
// counts another halving, so that c is 1 / 2 below 1, where the logarithm keeps its relative accuracy.  |r| < 2^-8, so
// the terms from r^4 on are carried in single precision.  Seven operations on the FP64 pipe against some twenty of log.
constexpr int kLogBits = 8, kLogHalf = 106, kLogTable = 2 << kLogBits;      // (c, -log c) pairs, then 34 values -e log 2
__device__ __forceinline__ double log_draw64(const double* __restrict__ table, uint32_t w) {
    const int k = 32 - __clz((int)w);                                       // 2 w + 1 = 2^k m
    const unsigned long long frac = (((unsigned long long)w << 1 | 1ull) << (52 - k)) & 0xfffffffffffffull;
    const double m = __longlong_as_double((long long)(frac | 0x3ff0000000000000ull));
    const int i = (int)(frac >> (52 - kLogBits));
    const double2 t = __ldg((const double2*)table + i);
    const double te = __ldg(table + kLogTable + (33 - k - (i >= kLogHalf ? 1 : 0)));
    const double r = fma(m, t.x, -1.0);
    const float rf = f32_trunc(r), q = fmaf(rf, fmaf(rf, fmaf(rf, 1.f / 7.f, -1.f / 6.f), 0.2f), -0.25f);
    const double p = fma(r, fma(r, f64_exact(q), 1.0 / 3.0), -0.5);
    return (te + t.y) + fma(r * r, p, r);
}
// sin and cos of 2 pi (w + 1/2) 2^-32: the nearest of 256 tabulated angles and the rest a, |a| < 0.0123, by the series of
// sin a and cos a - 1 (tails in single precision) and the addition theorems.  Fourteen operations on the FP64 pipe.
constexpr int kSinTable = kLogTable + 34, kDrawTable = kSinTable + 512;     // 256 (sin, cos) pairs after the logarithm's
__device__ __forceinline__ void sincos_draw64(const double* __restrict__ table, uint32_t w, double& sn, double& cs) {
    const double2 t = __ldg((const double2*)(table + kSinTable) + ((w + 0x800000u) >> 24));
    const int d = (int)(w << 8) >> 8;                                       // w less the tabulated angle's draw
    const double turn = __hiloint2double(0x41300000, d + 0x800000) - (1048576.0 + 0x1p-9);     // d 2^-32
    const double a = fma(turn, 6.283185307179586477, 7.314590396335798e-10), a2 = a * a;
    const float f = f32_trunc(a2);
    const double s = fma(a * a2, fma(a2, f64_exact(fmaf(f, -1.f / 5040.f, 1.f / 120.f)), -1.0 / 6.0), a);
    const double c = a2 * fma(a2, f64_exact(fmaf(f, -1.f / 720.f, 1.f / 24.f)), -0.5);
    sn = t.x + fma(t.y, s, t.x * c);
    cs = t.y + fma(-t.x, s, t.y * c);
}
inline void draw_table(double* table) {
    for (int i = 0; i < 1 << kLogBits; ++i) {
        const bool half = i >= kLogHalf;
        const double mid = 1.0 + (i + 0.5) / (1 << kLogBits), c = i + 1 == 1 << kLogBits ? 0.5 : std::rint(4096.0 / mid) / 4096.0;
        table[2 * i] = c;
        table[2 * i + 1] = -std::log(half ? 2.0 * c : c);
    }
    for (int e = 0; e < 34; ++e) table[kLogTable + e] = -e * 0.69314718055994530942;
    // the first octant's values, and the others by symmetry (exact zeros and ones on the axes)
    for (int j = 0; j < 256; ++j) {
        const int quarter = j >> 6, k = j & 63, o = k > 32 ? 64 - k : k;
        const double angle = o * (3.14159265358979323846 / 128.0), so = std::sin(angle), co = std::cos(angle);
        const double sk = k > 32 ? co : so, ck = k > 32 ? so : co;
        const double sv = quarter == 0 ? sk : quarter == 1 ? ck : quarter == 2 ? -sk : -ck;
        const double cv = quarter == 0 ? ck : quarter == 1 ? -sk : quarter == 2 ? -ck : sk;
        table[kSinTable + 2 * j] = sv;
        table[kSinTable + 2 * j + 1] = cv;
    }
}

// m and shift of a factor k > 0 for split_product64; shift 0: it has none
inline void factor64(double k, unsigned long long& m, int& shift) {
    int x = 0;
    const double f = std::frexp(k, &x);                  // k = f 2^x, f in [1/2, 1)
    m = (unsigned long long)std::ldexp(f, 53) << 11;
    shift = 51 - (x - 1);
    if (!(k > 0.0) || shift < 43 || shift > 75) { m = 0; shift = 0; }
}

}  // namespace phosim
