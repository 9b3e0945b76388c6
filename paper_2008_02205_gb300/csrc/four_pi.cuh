// v / (4 pi) rounded as the division rounds it, without dividing: q = v r with r = 1 / (4 pi)
// rounded, then one correction by the exact remainder v - 4 pi q, which rounds correctly
// (Markstein, Computation of elementary functions on the IBM RISC System/6000 processor, 1990).
// Three FP64 operations.  The remainder is exact while nothing underflows; the few values
// near the ends of FP64's range are divided.
// Plain C++ apart from the qualifiers, so that the CPU tests compile it too.
#pragma once

#include <math.h>
#include <string.h>

#include "widen.cuh"

namespace mlpg {

constexpr double kFourPi = 12.566370614359172953850573533118;

MLPG_HD double four_pi_quotient(double v) {
    constexpr double r = 1.0 / kFourPi;
    const double q = v * r;
    return fma(fma(-q, kFourPi, v), r, q);
}
#ifdef __CUDACC__
__host__ __device__ __noinline__   // the division's code and its registers stay out of the callers' loops
#endif
inline double four_pi_division(double v) { return v / kFourPi; }
MLPG_HD double div_four_pi(double v) {
    double out = four_pi_quotient(v);
#ifdef __CUDA_ARCH__
    const uint32_t e = ((uint32_t)__double2hiint(v) >> 20) & 0x7ffu;
#else
    uint64_t bits;
    memcpy(&bits, &v, 8);
    const uint32_t e = (uint32_t)(bits >> 52) & 0x7ffu;
#endif
    if (e - 100u > 1900u && v != 0.0) out = four_pi_division(v);   // below 2^-923, above 2^977, not finite
    return out;
}
// rounded to FP32, which has nothing below 2^-150 and above 2^128
MLPG_HD float div_four_pi_f(double v) {
    const float f = (float)four_pi_quotient(v);
    return f == f ? f : (float)v;   // an infinity (the remainder is NaN), a NaN
}

}  // namespace mlpg
