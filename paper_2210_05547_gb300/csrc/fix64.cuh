// Binary64 exponential, logarithm, quotient, reciprocal and roots on 64-bit integers.
//
// GB300 has one binary64 unit per SM: a warp-wide DFMA, DADD or DMUL holds it for 19 cycles
// (measured; 64 cycles from issue to result), while a 64 x 64 -> high 64 bit integer product
// takes 4 to 5 cycles of the SM's integer pipes, a 64-bit sum under 1 and a 32-bit product 0.5 to
// 1. The functions below therefore run entirely on integers, with 58 to 62 significant bits
// where binary64 carries 53, and round once when they return a binary64 value: they are cheaper
// and closer to the exact result than any binary64 sequence. The binary64 unit then runs the
// sums and products around them, at the same time.
//
// Everything here is plain integer arithmetic, the same on the host as on the device (the
// starting values of the reciprocal and root differ: the device takes the hardware's
// approximations, the host rounds exact ones to the same 23 bits).
#pragma once

#include <stdint.h>
#include <string.h>
#include <math.h>

#include "fix_table.h"

#ifdef __CUDACC__
#define FX __host__ __device__ __forceinline__
#else
#define FX static inline
#endif

namespace hyp {

typedef unsigned long long u64;
typedef long long i64;
typedef uint32_t u32;

#ifdef __CUDACC__
__device__ const u64 FIX_EXP_DEV[256] = {FIX_EXP_BODY};
__device__ const u64 FIX_LOG_DEV[128][2] = {FIX_LOG_BODY};
#endif
static const u64 FIX_EXP_HOST[256] = {FIX_EXP_BODY};
static const u64 FIX_LOG_HOST[128][2] = {FIX_LOG_BODY};

FX u64 fix_exp_entry(int j) {
#ifdef __CUDA_ARCH__
    return FIX_EXP_DEV[j];
#else
    return FIX_EXP_HOST[j];
#endif
}

FX const u64* fix_log_row(int j) {
#ifdef __CUDA_ARCH__
    return FIX_LOG_DEV[j];
#else
    return FIX_LOG_HOST[j];
#endif
}

FX u64 bits_of(double x) {
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(x);
#else
    u64 u;
    memcpy(&u, &x, 8);
    return u;
#endif
}

FX double double_of(u64 u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((i64)u);
#else
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}

FX int clz64(u64 x) {       // x != 0
#ifdef __CUDA_ARCH__
    return __clzll((i64)x);
#else
    return __builtin_clzll(x);
#endif
}

FX int clz32(u32 x) {       // x != 0
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return __builtin_clz(x);
#endif
}

FX u32 mulhi32(u32 a, u32 b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (u32)(((u64)a * b) >> 32);
#endif
}

FX int mulhi32s(int a, int b) {
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int)(((i64)a * b) >> 32);
#endif
}

// The high 64 bits of a b, at most two units low: the carry out of the low words is not formed
// (three 32-bit products instead of four and their carries).
FX u64 mulhi64(u64 a, u64 b) {
    const u32 ah = (u32)(a >> 32), al = (u32)a, bh = (u32)(b >> 32), bl = (u32)b;
    return (u64)ah * bh + mulhi32(ah, bl) + mulhi32(al, bh);
}

// The high 64 bits of a signed by an unsigned factor (a few units off).
FX i64 mulhi64su(i64 a, u64 b) {
    const u64 p = mulhi64((u64)a, b);
    return (i64)(a < 0 ? p - b : p);
}

// a b 2^-64 rounded to the nearest integer, a signed.
FX i64 mulhi64su_rn(i64 a, u64 b) {
    const u64 m = (u64)(a < 0 ? -a : a);
#ifdef __CUDA_ARCH__
    const u64 p = __umul64hi(m, b) + ((m * b) >> 63);
#else
    const unsigned __int128 w = (unsigned __int128)m * b;
    const u64 p = (u64)(w >> 64) + (u64)((w >> 63) & 1);
#endif
    return a < 0 ? -(i64)p : (i64)p;
}

// A positive number (m / 2^63) 2^e, m in [2^63, 2^64), or zero (m = 0).
struct xf {
    u64 m;
    int e;
};

FX xf xf_mul(xf a, xf b) {
    const u64 p = mulhi64(a.m, b.m);            // [2^62, 2^64)
    const int up = (int)(p >> 63);
    return xf{up ? p : p + p, a.e + b.e + up};
}

// The xf of a positive normal binary64 value.
FX xf xf_of(double x) {
    const u64 u = bits_of(x);
    return xf{(u << 11) | 0x8000000000000000ull, (int)((u >> 52) & 0x7ff) - 1023};
}

// v 2^-q (v any 64-bit value) normalised.
FX xf xf_fixed(u64 v, int q) {
    if (v == 0) return xf{0, 0};
    const int z = clz64(v);
    return xf{v << z, 63 - z - q};
}

// The binary64 nearest to x, for exponents inside binary64's normal range.
FX double f64_of_xf(xf x) {
    if (x.m == 0) return 0.0;
    const u64 v = (x.m >> 11) + ((x.m >> 10) & 1);      // leading one at bit 52, or 2^53 if carried
    return double_of(v + ((u64)(u32)(x.e + 1022) << 52));
}

// The same for any exponent: zero below the normal range, infinity above it.
FX double f64_of_xf_any(xf x) {
    if (x.m == 0 || x.e < -1022) return 0.0;
    if (x.e > 1022) return double_of(0x7ff0000000000000ull);
    return f64_of_xf(x);
}

FX double f64_of_fixed(u64 v, int q) { return f64_of_xf(xf_fixed(v, q)); }

FX float rcp_start(float x) {      // 1 / x within 2^-22, x in [1, 2)
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;
#endif
}

FX float rsqrt_start(float x) {    // 1 / sqrt(x) within 2^-22, x in [1, 4)
#ifdef __CUDA_ARCH__
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / sqrtf(x);
#endif
}

FX float float_of_bits(u32 u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x;
    memcpy(&x, &u, 4);
    return x;
#endif
}

FX u32 bits_of_float(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    u32 u;
    memcpy(&u, &x, 4);
    return u;
#endif
}

// 2^127 / m for m in [2^63, 2^64): the reciprocal of a mantissa as a mantissa of the same form
// (2 ulp of 2^-62; just below 2^64 for m = 2^63). A start y of 23 bits and one third-order step
// y (1 + d + d^2) with the residual d = 1 - m y exact to 2^-63: the error d^3 is below 2^-62.
FX u64 rcp64(u64 m) {
    const float f = float_of_bits(0x3f800000u | (u32)((m >> 40) & 0x7fffffu));    // [1, 2)
    // the start in (1/2, 1], lowered by 2^-22 so that it stays below 1, as y 2^-32
    const float y0 = rcp_start(f);
    const u32 b = bits_of_float(y0);                     // exponent 126 (or 127 for y0 = 1)
    const u32 y = b >= 0x3f800000u ? 0xfffffc00u : (((b & 0x7fffffu) | 0x800000u) << 8) - 0x400u;
    // m y with m = f 2^63: f y = 1 - d, in units of 2^-63
    const u64 p = (u64)(u32)(m >> 32) * y + mulhi32((u32)m, y);
    // (p is up to one low; one less keeps the result below 2^64 at m = 2^63)
    const i64 d = (i64)(0x7fffffffffffffffull - p);      // |d| < 2^42
    const int dh = (int)(d >> 12);                       // units of 2^-51
    const u64 c = (u64)(d + (i64)(((i64)dh * dh) >> 39)); // d + d^2, units of 2^-63
    // y (1 + c) in units of 2^-64, then the mantissa in [2^63, 2^64)
    const i64 yc = (i64)((i64)(int)(c >> 31) * (i64)y) + (i64)(((u64)(u32)(c & 0x7fffffffu) * y) >> 31);
    return ((u64)y << 32) + (u64)yc;
}

FX xf xf_rcp(xf a) { return xf{rcp64(a.m), -a.e - 1}; }

// 2^64 / sqrt(f) for f = m 2^-62 in [1, 4), m in [2^62, 2^64): the mantissa of the reciprocal root,
// value r 2^-64. A 23-bit start and one third-order step y (1 + d/2 + 3/8 d^2), d = 1 - f y^2.
FX u64 rsqrt64(u64 m) {
    const int up = (int)(m >> 63);                       // f >= 2
    const float f = float_of_bits((up ? 0x40000000u : 0x3f800000u) |
                                  ((u32)(m >> (up ? 40 : 39)) & 0x7fffffu));
    const u32 b = bits_of_float(rsqrt_start(f));
    const u32 y = b >= 0x3f800000u ? 0xfffffc00u : (((b & 0x7fffffu) | 0x800000u) << 8) - 0x400u;
    const u64 p = mulhi64(m, (u64)y * y);                // f y^2 in units of 2^-62, up to 2 low
    const i64 d = (i64)(0x3fffffffffffffffull - p);      // |d| < 2^43
    const int dh = (int)(d >> 12);                       // units of 2^-50
    const u64 c = (u64)(d + ((3 * ((i64)dh * dh)) >> 40));   // d/2 + 3/8 d^2, units of 2^-63
    const i64 yc = (i64)((i64)(int)(c >> 31) * (i64)y) + (i64)(((u64)(u32)(c & 0x7fffffffu) * y) >> 31);
    return ((u64)y << 32) + (u64)yc;
}

// e^a for a reduction already split off: a = kk ln2/256 + r, r72 = r in units of 2^-72
// (0 <= r < 1.02 ln2/256). 2^(kk / 256) from the table times 1 + r + r^2/2 + r^3 (1/6 + r/24 +
// r^2/120), the terms from the third on in 32-bit words; about 2^-58 of the value.
FX xf exp_reduced(int kk, u64 r72) {
    const u64 t = fix_exp_entry(kk & 255);               // 2^-62
    const u64 r2 = mulhi64(r72, r72);                    // r^2, 2^-80
    const u32 rh = (u32)(r72 >> 32);                     // 2^-40
    const u32 r3 = mulhi32((u32)(r2 >> 32), rh);         // r^3, 2^-56
    // 1/6 + r/24 + r^2/120 in units of 2^-34
    const u32 c = 2863311531u + mulhi32(rh, 2796203u + mulhi32(rh, 2185u));
    const u64 p = r72 + (r2 >> 9) + (((u64)r3 * c) >> 18);   // e^r - 1, 2^-72
    const u64 v = t + (mulhi64(t, p) >> 8);              // [1, 2.0001) in units of 2^-62
    const int up = (int)(v >> 63);
    return xf{up ? v : v + v, (kk >> 8) + up};
}

// e^a, a in units of 2^-Q (Q 53: |a| < 1023; Q 58: |a| < 32).
template <int Q>
FX xf exp_fixed(i64 a) {
    // floor(a 256/ln2), at most 0.01 low: the residue stays nonnegative
    const int kk = (mulhi32s((int)(a >> 32), FIX_EXP_K19 >> (Q - 53)) - 1) >> 8;
    const u64 r72 = ((u64)a << (72 - Q)) - (u64)(i64)kk * FIX_EXP_C72;
    return exp_reduced(kk, r72);
}

// e^x for a finite binary64 |x| < 512 (the caller checks): the reduction takes every bit of x.
FX double fix_exp(double x) {
    const u64 u = bits_of(x);
    const int ex = (int)((u >> 52) & 0x7ff) - 1023;      // < 9
    const u64 m = (u << 11) | 0x8000000000000000ull;     // |x| 2^(63 - ex)
    const bool neg = (i64)u < 0;
    // |x| in units of 2^-72 mod 2^64 and its leading part in units of 2^-21
    const int s = 9 + ex;
    u64 a72 = s >= 0 ? m << s : (s > -64 ? m >> -s : 0);
    const int sh = 10 - ex;
    int ah = sh < 32 ? (int)((u32)(m >> 32) >> sh) : 0;
    if (neg) {
        a72 = 0 - a72;
        ah = -ah - 1;
    }
    const int kk = (mulhi32s(ah, FIX_EXP_K19) - 1) >> 8;
    return f64_of_xf(exp_reduced(kk, a72 - (u64)(i64)kk * FIX_EXP_C72));
}

// ln x in units of 2^-58 for a normal x in [2^-45, 2^45]: x = 2^k y, y in [1, 2), j the top 7
// fraction bits of y, r = y inv_j - 1 (|r| < 2^-8), ln x = k ln2 - ln inv_j + log1p(r); within
// 2^-54.
FX i64 log58(double x) {
    const u64 u = bits_of(x);
    const int k = (int)((u >> 52) & 0x7ff) - 1023;
    const u64 m = (u << 11) | 0x8000000000000000ull;
    const u64* row = fix_log_row((int)(m >> 56) & 127);
    const i64 r = (i64)(mulhi64(m, row[0]) - 0x8000000000000000ull);   // 2^-63, |r| < 2^55
    const i64 rs = r << 7;                               // 2^-70
    const int rh = (int)(rs >> 32);                      // 2^-38
    const u64 ra = (u64)(rs < 0 ? -rs : rs);
    const u64 r2 = mulhi64(ra, ra);                      // 2^-76
    // 1/3 - r/4 + r^2/5 - r^3/6 + r^4/7 in units of 2^-32 (r/4 and on from 32-bit words)
    const int c3 = 715827883 - (int)mulhi32s(rh, 9586981);   // 1/6 - r/7, units of 2^-32
    const int c2 = 858993459 - (mulhi32s(rh, c3) >> 6);      // 1/5 - r (...)
    const int c1 = 1073741824 - (mulhi32s(rh, c2) >> 6);     // 1/4 - r (...)
    const int c0 = 1431655765 - (mulhi32s(rh, c1) >> 6);     // 1/3 - r (...)
    const int r3 = (int)(((i64)(int)(r2 >> 29) * rh) >> 31);   // r^3, 2^-54
    const i64 l = (r >> 5) - (i64)(r2 >> 19) + (((i64)r3 * c0) >> 28);   // log1p(r), 2^-58
    return (i64)k * (i64)FIX_LN2_58 + (i64)row[1] + l;
}

// The binary64 nearest to v 2^-q for a signed v (the sign set in its bit: a negation would issue on
// the binary64 pipe).
FX double f64_of_signed(i64 v, int q) {
    const double x = f64_of_fixed((u64)(v < 0 ? -v : v), q);
    return double_of(bits_of(x) | ((u64)v & 0x8000000000000000ull));
}

// ---- fixed-point numbers of a common scale (line solver, filters): values below 2^E in magnitude ----

// m >> s, zero for s outside 0..63.
FX u64 shift_down(u64 m, int s) {
#ifdef __CUDA_ARCH__
    u64 v;
    asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(s));   // PTX clamps the shift amount
    return v;
#else
    return (unsigned)s < 64u ? m >> s : 0;
#endif
}

FX int high_word(double x) { return (int)(bits_of(x) >> 32); }
FX unsigned magnitude(double x) { return (unsigned)high_word(x) & 0x7fffffffu; }   // of |x|
FX unsigned larger(unsigned a, unsigned b) { return a > b ? a : b; }

// Values whose largest high word is `top`: too large (or not finite) for a common scale, or its E.
FX bool scale_wild(unsigned top) { return top >= (unsigned)(1023 + 899) << 20; }
FX int scale_of(unsigned top) {
    const int E = (int)(top >> 20) - 1022;
    return E > -960 ? E : -960;
}

// Whether values whose largest high word is `top` are zero or have a scale of their own (E above its
// floor of -960, below which units of 2^(E - 62) would leave binary64's normal range).
FX bool scale_fits(unsigned top) {
    return top == 0u || (!scale_wild(top) && top >= (unsigned)(1023 - 960) << 20);
}

// x in units of 2^(E - q), truncated towards zero.
FX i64 to_scale(double x, int E, int q) {
    const int hi = high_word(x);
    const u64 m = (bits_of(x) << 11) | 0x8000000000000000ull;
    const i64 v = (i64)shift_down(m, 63 - q + E + 1023 - ((hi >> 20) & 0x7ff));
    const i64 s = hi >> 31;
    return (v ^ s) - s;
}

// The binary64 nearest to m 2^(E - q) for m < 2^33, its sign bit set by `sign`.
#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
inline double small_from_scale(u64 m, int E, int q, unsigned sign) {
    return double_of(bits_of(f64_of_fixed(m, q - E)) | (u64)sign << 32);
}

// The binary64 nearest to y 2^(E - q), |y| < 2^63, its sign flipped by `sign` (0 or the sign bit).
FX double from_scale(i64 y, int E, int q, unsigned sign = 0) {
    const int s = (int)(y >> 63);
    const u64 m = (u64)((y ^ (i64)s) - (i64)s);
    const u32 h = (u32)(m >> 32);
    const unsigned sg = ((unsigned)s & 0x80000000u) ^ sign;
    if (h < 2u) return small_from_scale(m, E, q, sg);
    const int z = clz32(h) - 1;                          // leading one to bit 62
    const u64 v = ((m << z) + 0x200) >> 10;              // [2^52, 2^53]
    return double_of((v + ((u64)(u32)(E + 62 - q - z + 1022) << 52)) | (u64)sg << 32);
}

// a c 2^-64 for a constant c = h 2^32 + l (h >= 0), |a| h and |a| l small enough that the sum of
// cross products stays below 2^63.
FX i64 mul_const(i64 a, int h, int l) {
    const int ah = (int)(a >> 32);
    const i64 x = (i64)ah * l + (i64)((u64)(u32)a * (u32)h);
    return (i64)ah * h + (x >> 32);
}

constexpr int RUN = 4;                                   // outputs per thread of the filters and differences

// Tenth differences over 1024 (weights 252, -210, 120, -45, 10, -1) of the four windows of eleven in
// x, in 72 bits (high and low words apart) and so within 2 units of 2^-62 of the largest input; then
// rounded to binary64. False where that is not better than binary64: inputs that are not finite, huge
// or tiny, or a window whose inputs may all be below 2^-7 of the largest.
FX bool tenth_run(const double (&x)[RUN + 10], double (&acc)[RUN]) {
    unsigned core = 0, ends = 0;                         // core: in every window
    for (int k = 0; k < RUN + 10; ++k) {
        if (k >= RUN - 1 && k < 11) core = larger(core, magnitude(x[k]));
        else ends = larger(ends, magnitude(x[k]));
    }
    const unsigned top = larger(core, ends);
    if (!scale_fits(top) || (core >> 20) + 6 < top >> 20) return false;
    const int E = scale_of(top);
    i64 v[RUN + 10];
#pragma unroll
    for (int k = 0; k < RUN + 10; ++k) v[k] = to_scale(x[k], E, 62);
#pragma unroll
    for (int o = 0; o < RUN; ++o) {
        const i64 s[6] = {v[o + 5], v[o + 4] + v[o + 6], v[o + 3] + v[o + 7], v[o + 2] + v[o + 8],
                          v[o + 1] + v[o + 9], v[o] + v[o + 10]};
        const u32 w[6] = {252, 210, 120, 45, 10, 1};
        i64 h = 0;
        u64 even = 0, odd = 0;                           // low words' sums
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            h += (i64)(int)(s[k] >> 32) * (k & 1 ? -(int)w[k] : (int)w[k]);
            (k & 1 ? odd : even) += (u64)(u32)s[k] * w[k];
        }
        acc[o] = from_scale((h << 22) + ((i64)(even - odd) >> 10), E, 62);
    }
    return true;
}

FX i64 fourth_difference(i64 a, i64 b, i64 c, i64 d, i64 e) { return (a + e) - 4 * (b + d) + 6 * c; }

// sums[k] = d4x wt[0] + d4y wt[1] of four neighbours, the fourth differences along their row w (two
// before to two after) and across it over the rows r (two below, one below, one above, two above).
// Sixteen units of 2^-59 of the power of two above the largest of the 24 inputs bound the error of
// either difference; false where that may exceed binary64's
// (rms 2^-52.2 of the largest of a difference's five inputs, here 2^-52.7 at the line drawn): an
// output one of whose two windows lies below 2^-5 of the largest, or inputs not finite, huge or tiny.
FX bool fourth_run(const double (&w)[RUN + 4], const double (&r)[4][RUN], const double (&wt)[2],
                   double (&sums)[RUN]) {
    unsigned mw[RUN + 4], top = 0, least = ~0u;
#pragma unroll
    for (int k = 0; k < RUN + 4; ++k) mw[k] = magnitude(w[k]);
    const unsigned mid = larger(mw[3], mw[4]);
#pragma unroll
    for (int k = 0; k < RUN; ++k) {
        unsigned mx = mid, my = mw[k + 2];
#pragma unroll
        for (int q = 0; q < 5; ++q)
            if (k + q != 3 && k + q != 4) mx = larger(mx, mw[k + q]);
#pragma unroll
        for (int q = 0; q < 4; ++q) my = larger(my, magnitude(r[q][k]));
        const unsigned lo = mx < my ? mx : my;
        top = larger(top, larger(mx, my));
        least = lo < least ? lo : least;
    }
    if (!scale_fits(top) || (least >> 20) + 4 < top >> 20) return false;
    const int E = scale_of(top);
    i64 v[RUN + 4];
#pragma unroll
    for (int k = 0; k < RUN + 4; ++k) v[k] = to_scale(w[k], E, 59);
#pragma unroll
    for (int k = 0; k < RUN; ++k) {
        const double dx = from_scale(fourth_difference(v[k], v[k + 1], v[k + 2], v[k + 3], v[k + 4]), E, 59);
        sums[k] = fma(from_scale(fourth_difference(to_scale(r[0][k], E, 59), to_scale(r[1][k], E, 59), v[k + 2],
                                                   to_scale(r[2][k], E, 59), to_scale(r[3][k], E, 59)), E, 59),
                      wt[1], dx * wt[0]);
    }
    return true;
}

// Four outputs of the nine-point Gaussian filter over the windows of nine in x, within 11 units of 2^-62 of the run's
// power of two before their rounding. Returns the mask of outputs for which that is not better than
// binary64 (above 2^-53.5 of the output, or inputs that are not finite, huge or tiny).
FX int gauss_fixed(const double (&x)[RUN + 8], double (&y)[RUN]) {
    // the weights (centre, +-1, .. +-4) in units of 2^-64, as the words (h, l) of mul_const
    const int wh[5] = {1476809260, 1024362956, 330904695, 49378868, 4432499};
    const int wl[5] = {1060485752, 721130311, -710525454, -721130311, 180282578};
    unsigned top = 0;
#pragma unroll
    for (int k = 0; k < RUN + 8; ++k) top = larger(top, magnitude(x[k]));
    if (!scale_fits(top)) return (1 << RUN) - 1;
    const int E = scale_of(top);
    i64 v[RUN + 8];
#pragma unroll
    for (int k = 0; k < RUN + 8; ++k) v[k] = to_scale(x[k], E, 62);
    int coarse = 0;
#pragma unroll
    for (int o = 0; o < RUN; ++o) {
        i64 acc = mul_const(v[o + 4], wh[0], wl[0]);
#pragma unroll
        for (int d = 1; d <= 4; ++d)
            acc += mul_const(v[o + 4 - d] + v[o + 4 + d], wh[d], wl[d]);
        y[o] = from_scale(acc, E, 62);
        const int h = (int)(acc >> 32);
        if ((u32)(h ^ (h >> 31)) < 1u << 25) coarse |= 1 << o;   // |acc| < 2^57
    }
    return top == 0u ? 0 : coarse;
}

// 1 / b, a / b, sqrt(a) and 1 / sqrt(a) for b in [2^-500, 2^500] in magnitude and a of the same range
// (positive under the roots): one rounding, within 0.51 ulp.
FX double fix_rcp(double b) {
    const u64 u = bits_of(b);
    const double r = f64_of_xf(xf_rcp(xf_of(b)));
    return double_of(bits_of(r) | (u & 0x8000000000000000ull));
}

FX double fix_div(double a, double b) {
    const u64 s = (bits_of(a) ^ bits_of(b)) & 0x8000000000000000ull;
    const double q = f64_of_xf(xf_mul(xf_of(a), xf_rcp(xf_of(b))));
    return double_of(bits_of(q) | s);
}

FX xf xf_rsqrt(xf a) {
    const int odd = a.e & 1;                             // f = (m / 2^63) 2^odd in [1, 4)
    const u64 r = rsqrt64(odd ? a.m : a.m >> 1);
    return xf{r, -((a.e - odd) >> 1) - 1};
}

FX double fix_rsqrt(double a) { return f64_of_xf(xf_rsqrt(xf_of(a))); }

FX double fix_sqrt(double a) {
    const xf x = xf_of(a);
    return f64_of_xf(xf_mul(x, xf_rsqrt(x)));
}

}  // namespace hyp
