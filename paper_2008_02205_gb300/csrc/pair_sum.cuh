// Sums of FP32 values in unevaluated pairs of floats (hi + lo): the two-sum of Knuth (The Art
// of Computer Programming, vol. 2, 4.2.2, theorem B) gives the rounding error of hi + x
// exactly, lo collects those errors.  48 bits, where a sum of floats has 24: for
// the partial sums of FP32 dot products, which the FP64 units (1.6 additions per clock and
// SM) would bound.  Plain C++ apart from the qualifiers and the intrinsics that keep the
// compiler from contracting, so that the CPU tests compile it too.
#pragma once

#include "widen.cuh"

namespace mlpg {

#ifdef __CUDA_ARCH__
MLPG_HD float add_rn(float a, float b) { return __fadd_rn(a, b); }
MLPG_HD float mul_rn(float a, float b) { return __fmul_rn(a, b); }
#else
MLPG_HD float add_rn(float a, float b) { return a + b; }
MLPG_HD float mul_rn(float a, float b) { return a * b; }
#endif

// what a thread sums products of vector values in: FP64 for FP64, a pair for FP32
template <typename T>
struct Sum {   // T = double
    double v;
    MLPG_HD void clear() { v = 0.0; }
    MLPG_HD void add_product(double a, double b) { v += a * b; }
    MLPG_HD void add(const Sum &o) { v += o.v; }
    MLPG_HD double value() const { return v; }
};
template <>
struct Sum<float> {
    float hi, lo;
    MLPG_HD void clear() { hi = lo = 0.0f; }
    MLPG_HD void add(float x) {
        const float s = add_rn(hi, x), b = add_rn(s, -hi);
        lo = add_rn(lo, add_rn(add_rn(hi, -add_rn(s, -b)), add_rn(x, -b)));
        hi = s;
    }
    MLPG_HD void add_product(float a, float b) { add(mul_rn(a, b)); }
    MLPG_HD void add(const Sum &o) {
        add(o.hi);
        lo = add_rn(lo, o.lo);
    }
    MLPG_HD double value() const { return (double)hi + (double)lo; }
};

// The same with three floats: the errors of lo's additions go on into a third, so that a sum of floats
// is held in more than the 53 bits of an FP64 sum.
struct TripleSum {
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
    MLPG_HD static float two_sum(float &s, float x) {   // s += x; returns the rounding error
        const float a = s, b = add_rn(add_rn(a, x), -a);
        s = add_rn(a, x);
        return add_rn(add_rn(a, -add_rn(s, -b)), add_rn(x, -b));
    }
    MLPG_HD void add(float x) { lo = add_rn(lo, two_sum(mid, two_sum(hi, x))); }
    MLPG_HD double value() const { return (double)hi + ((double)mid + (double)lo); }
};

}  // namespace mlpg
