// FP32 -> FP64 by integer moves, for kernels that the FP64 units bound: the conversion
// runs on those units, at 1.9 per clock and SM, and costs as much as the multiply-add or
// addition that follows it; the ten integer instructions here run beside them.
// Exact for every FP32 value, subnormals, infinities and NaNs included.
// Plain C++ apart from the qualifiers, so that the CPU tests compile it too.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MLPG_HD __host__ __device__ __forceinline__
#else
#define MLPG_HD inline
#endif

namespace mlpg {

// high and low word of the double that equals the float with bits b
MLPG_HD void widen_words(uint32_t b, uint32_t &hi, uint32_t &lo) {
    const uint32_t t = b & 0x7fffffffu;
#ifdef __CUDA_ARCH__
    const int lead = __clz((int)t);
#else
    const int lead = t ? __builtin_clz(t) : 32;
#endif
    const int sh = t < 0x00800000u ? lead - 8 : 0;   // a subnormal's leading bit to the implicit one's place
    const uint32_t m = t << sh;                      // exponent field (1 for a subnormal) and mantissa
    uint32_t h = (m >> 3) + ((uint32_t)(1023 - 127 - sh) << 20);
    if (t >= 0x7f800000u) h += (uint32_t)(2047 - 255 - (1023 - 127)) << 20;   // infinity, NaN
    if (t == 0) h = 0;
    hi = h | (b & 0x80000000u);
    lo = m << 29;
}

}  // namespace mlpg
