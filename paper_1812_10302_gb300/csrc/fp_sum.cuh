// fp_sum.cuh -- sums of FP32 values and squares, exact to well past FP64, in
// FP32 arithmetic with error-free transformations (this part issues FP64 at
// 1/64 of its FP32 rate).
#pragma once

#include <cuda_runtime.h>

namespace dtws {

// A running sum of three floats a + b + c; a and b are updated by TwoSum
// (Knuth), so only c rounds (second-order compensated summation, Klein 2006):
// n terms are exact to about n^2 2^-72 of the largest partial sum.  The
// intrinsics keep the compiler from contracting a product and a sum.
struct f3 {
    float a, b, c;
};
struct exact2 {
    float s, e;
};
__device__ __forceinline__ exact2 two_sum_rn(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
// t += h + l
__device__ __forceinline__ void f3_add(f3 &t, float h, float l) {
    const exact2 p = two_sum_rn(t.a, h), q = two_sum_rn(t.b, l), r = two_sum_rn(q.s, p.e);
    t.a = p.s;
    t.b = r.s;
    t.c = __fadd_rn(t.c, __fadd_rn(q.e, r.e));
}
// t += (h + l)^2
__device__ __forceinline__ void f3_add_sq(f3 &t, float h, float l) {
    const float p = __fmul_rn(h, h), pe = __fmaf_rn(h, h, -p);
    const float h2 = __fadd_rn(h, h), q = __fmul_rn(h2, l), qe = __fmaf_rn(h2, l, -q);
    f3_add(t, p, pe);
    const exact2 r = two_sum_rn(t.b, q);
    t.b = r.s;
    t.c = __fadd_rn(t.c, __fadd_rn(r.e, __fmaf_rn(l, l, qe)));
}
__device__ __forceinline__ double f3_value(const f3 &t) { return ((double)t.c + (double)t.b) + (double)t.a; }

// Mean (FP64) and variance of n samples y over `threads` threads' shares
// (start t, stride `threads`): each thread's part is summed in FP32 expansions,
// the parts in FP64 by `reduce` (the same result in every thread) -- two-pass,
// no less exact than FP64 sums throughout and not bound by this part's FP64
// rate.  Sums that overflow FP32 are taken again on samples scaled by 2^-80.
// (None underflows that matters: a variance below 1e-24 counts as none.)
template <typename Reduce>
__device__ __forceinline__ void mean_and_variance(const float *__restrict__ y, int n, int t, int threads, Reduce &&reduce,
                                                  double &mu, double &var) {
    float f = 1.0f;
    for (;;) {
        f3 s{0.0f, 0.0f, 0.0f};
        for (int j = t; j < n; j += threads) f3_add(s, __fmul_rn(y[j], f), 0.0f);
        mu = reduce(f3_value(s)) / (double)n;
        const float mh = (float)mu, ml = (float)(mu - (double)mh);
        f3 v{0.0f, 0.0f, 0.0f};
        for (int j = t; j < n; j += threads) {
            exact2 d = two_sum_rn(__fmul_rn(y[j], f), -mh);
            d = two_sum_rn(d.s, __fsub_rn(d.e, ml));
            f3_add_sq(v, d.s, d.e);
        }
        var = reduce(f3_value(v)) / (double)n;
        if (isfinite(var) || f < 1.0f) break;
        f = 0x1p-80f;
    }
    mu *= f < 1.0f ? 0x1p80 : 1.0;
    var *= f < 1.0f ? 0x1p160 : 1.0;
}

}  // namespace dtws
