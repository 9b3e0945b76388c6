// Sums of products in fixed point, for the pair sums of the integration: the FP64
// units do 1.6 operations per clock and SM, the integer multiplier some 30 wide
// products, and three of those (high x high, and the two mixed ones) stand for one
// FP64 multiply-add.
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
// e with |v| < 2^e for every value, from the largest high word (sign bit off); 0 for all zeros
__device__ __forceinline__ int top_exp(unsigned hiword) { return hiword ? (int)(hiword >> 20) - 1022 : 0; }

}  // namespace
}  // namespace mlpg
