// The closure's binary64 exponential, logarithm, quotient, reciprocal and roots: the integer forms
// of fix64.cuh inside their ranges, CUDA's own functions outside.
//
// In FP64 instructions (19 cycles of the SM's one binary64 unit per warp), CUDA's exp issues 15,
// log 28, a division 8, a reciprocal 5; table-driven binary64 forms (Tang 1989, 1990; Newton
// quotients), used here before, 7, 11, 5 and 4. The integer forms issue none: about 35, 30, 30 and
// 25 cycles of the integer pipes, beside the binary64 unit instead of on it, and they round once
// (0.6 ulp for exp, 0.51 for the others, against 2 and 1).
#pragma once

#include <cuda_runtime.h>

#include "fix64.cuh"
#include "fp32.cuh"

namespace hyp {

__device__ __forceinline__ int exponent_of(double x) {
    return ((__double2hiint(x) >> 20) & 0x7ff) - 1023;
}

// exp(x) within 1 ulp; |x| >= 512, NaN and infinities take CUDA's exp.
__device__ __forceinline__ double fast_exp(double x) {
    if (exponent_of(x) >= 9) return exp(x);
    return fix_exp(x);
}

// |b| in (2^-120, 2^120): the reciprocal's and divisor's range. Outside it, and for zero, NaN and
// infinities, CUDA's division.
__device__ __forceinline__ bool rcp_fast_range(double b) {
    return (unsigned)(exponent_of(b) + 119) < 239u;
}

__device__ __forceinline__ double fast_rcp(double b) {
    if (!rcp_fast_range(b)) return 1.0 / b;
    return fix_rcp(b);
}

// a / b within 1 ulp, a zero or in [2^-499, 2^500): the quotient then stays a normal number.
__device__ __forceinline__ double fast_div(double a, double b) {
    if (!rcp_fast_range(b)) return a / b;
    if ((unsigned)(exponent_of(a) + 499) >= 999u)
        return (bits_of(a) << 1) == 0 ? double_of((bits_of(a) ^ bits_of(b)) & (1ull << 63)) : a / b;
    return fix_div(a, b);
}

// log(x) within 1 ulp for x in [2, 2^45); CUDA's log otherwise (below 2 log x may be near zero,
// where the fixed-point result would lose relative accuracy).
__device__ __forceinline__ double fast_log(double x) {
    const int hx = __double2hiint(x);
    if (hx < 0x40000000 || hx >= 0x42c00000) return log(x);
    return f64_of_fixed((u64)log58(x), 58);
}

// 1 / sqrt(x) and sqrt(x) within 1 ulp for x in [2^-499, 2^500); CUDA's otherwise.
__device__ __forceinline__ double fast_rsqrt(double x) {
    if (__double2hiint(x) < 0 || (unsigned)(exponent_of(x) + 499) >= 999u) return rsqrt(x);
    return fix_rsqrt(x);
}

__device__ __forceinline__ double fast_sqrt(double x) {
    if (__double2hiint(x) < 0 || (unsigned)(exponent_of(x) + 499) >= 999u) return sqrt(x);
    return fix_sqrt(x);
}

}  // namespace hyp
