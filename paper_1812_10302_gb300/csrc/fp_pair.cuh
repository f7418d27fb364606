// fp_pair.cuh -- unevaluated sums of two floats.  (Plain C++ outside nvcc, where
// products and sums must not be contracted.)
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define DTWS_HD __host__ __device__ __forceinline__
#else
#define DTWS_HD inline
#endif

namespace dtws {

// Unevaluated sums hi + lo of two floats with error-free transformations
// (Knuth's TwoSum, Dekker's Fast2Sum, the FMA product error).
struct f2 {
    float hi, lo;
};
DTWS_HD f2 two_sum(float a, float b) {
    const float s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
DTWS_HD f2 fast_two_sum(float a, float b) {
    const float s = a + b;
    return {s, b - (s - a)};
}
DTWS_HD f2 f2_add(f2 x, f2 y) {
    f2 s = two_sum(x.hi, y.hi);
    const f2 t = two_sum(x.lo, y.lo);
    s.lo += t.hi;
    s = fast_two_sum(s.hi, s.lo);
    s.lo += t.lo;
    return fast_two_sum(s.hi, s.lo);
}
DTWS_HD f2 f2_neg(f2 x) { return {-x.hi, -x.lo}; }
DTWS_HD f2 f2_mul(f2 x, f2 y) {
    const float p = x.hi * y.hi;
    float e = fmaf(x.hi, y.hi, -p);
    e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, e));
    return fast_two_sum(p, e);
}
DTWS_HD f2 f2_mul_f(f2 x, float f) {
    const float p = x.hi * f;
    const float e = fmaf(x.lo, f, fmaf(x.hi, f, -p));
    return fast_two_sum(p, e);
}
// x - y, the low parts' difference rounded.  err bounds, in units of 2^-48,
// its distance from X - Y, the real numbers that x and y store (a pair is its
// number to 2^-49): half a unit of each, and 2^-24 of the two sums that are
// rounded, as they came out (bounded beforehand they would count two units of
// each number, twice what they are on average).  The last step is exact: where
// the high parts nearly cancel their difference is zero or no smaller than the
// low parts'.
DTWS_HD f2 f2_diff(f2 x, f2 y, float &err) {
    const f2 s = two_sum(x.hi, -y.hi);
    const float t = x.lo - y.lo, u = s.lo + t;
    err = fmaf(fabsf(t) + fabsf(u), 0x1p24f, 0.5f * (fabsf(x.hi) + fabsf(y.hi)));
    return fast_two_sum(s.hi, u);
}

}  // namespace dtws
