// Sums of products in fixed point, for the pair sums of the integration: the FP64
// units do 1.6 operations per clock and SM, the integer multiplier some 30 wide
// products, and three of those (high x high, and the two mixed ones) stand for one
// FP64 multiply-add.  Each function has its own scale, so that a pair's error is 2^-53 of the two
// functions' own largest values, whatever other functions share their points.
#pragma once

#include <stdint.h>

namespace mlpg {
namespace {
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
// v scale rounded to an integer of at most 56 bits, in two signed parts: hi 2^28 + lo, |lo| <= 2^27
__device__ __forceinline__ int2 fixed_parts(double v, double scale) {
    const long long x = __double2ll_rn(v * scale);
    const int lo = (int)((unsigned)x << 4) >> 4;
    return make_int2((int)((x - lo) >> 28), lo);
}
// e with |v| < 2^e for every value, from the largest high word (sign bit off); 0 for all zeros.  At least
// -900, so that the scale 2^(bits - e) is finite.
__device__ __forceinline__ int top_exp(unsigned hiword) { return hiword ? max((int)(hiword >> 20) - 1022, -900) : 0; }
__device__ __forceinline__ unsigned abs_hiword(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __noinline__ double pow2_subnormal(int k) { return ldexp(1.0, k); }
__device__ __forceinline__ double pow2(int k) {
    return (unsigned)(k + 1022) < 2046u ? __hiloint2double((k + 1023) << 20, 0) : pow2_subnormal(k);
}

}  // namespace
}  // namespace mlpg
