// series_kernels.cu -- per-series and per-(series, m | r) kernels:
//   * one pass over the series: finiteness check, largest |x| and in-block
//     excursion, its every fourth sample, level 0 of the block envelope;
//   * anchored, compensated prefix sums of the series (once per series),
//     stored as FP32 pairs;
//   * window statistics for a query length m (Sec. 2.2, Eq. 5, population
//     sigma) from those sums;
//   * the raw sliding envelope of the series for a band half-width r
//     (Sec. 2.2, Eq. 9 applied to the series, clipped to [0, n)).
#include <cmath>

#include "dtws_internal.h"
#include "fp_pair.cuh"
#include "fp_sum.cuh"

namespace dtws {

// ------------------------------------------------------------------ first pass
// One CTA per block of kBlockB samples reads the series once and takes from
// it everything that needs no other block: the finiteness flag, the largest
// |x| (as its FP32 bit pattern, which orders like the value for non-negative
// floats; meaningful when no value is NaN or Inf), the largest in-block
// excursion |x - x[block start]| (the scale of the prefix sums), the series'
// every kProxyStride-th sample (x_sub[j] = x[kProxyStride j]) and level 0 of
// the block envelope (max and min of kEnvG samples).  Bound by memory: 4 B
// read and 1.5 B written per sample.  (As four kernels, each reading the
// series again, the same work took 85 us per 1e7 samples.)
// x is the padded series, so whole float4s are read past n; those samples
// count for nothing.
constexpr int kFirstThreads = 256;
__global__ void __launch_bounds__(kFirstThreads)
k_series_first(const float *__restrict__ x, int64_t n, int *__restrict__ flag, unsigned *__restrict__ absmax,
               unsigned *__restrict__ excursion, float *__restrict__ x_sub, float *__restrict__ mx0,
               float *__restrict__ mn0, int64_t nblk) {
    static_assert(kProxyStride == 4 && kEnvG == 16, "one float4 per kept sample, four per envelope block");
    const int64_t t0 = (int64_t)blockIdx.x * kBlockB;
    const float inf = __int_as_float(0x7f800000);
    const float a = x[t0];
    const float4 *x4 = reinterpret_cast<const float4 *>(x + t0);
    bool bad = false;
    float amax = 0.0f, emax = 0.0f;
    // (a block's float4s: kBlockB / 4 = 8 per thread)
#pragma unroll
    for (int q = 0; q < kBlockB / 4 / kFirstThreads; ++q) {
        const int i = q * kFirstThreads + (int)threadIdx.x;
        const int64_t t = t0 + 4 * (int64_t)i;
        const float4 v = x4[i];
        const float w[4] = {v.x, v.y, v.z, v.w};
        float hi = -inf, lo = inf;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (t + e < n) {
                bad |= !isfinite(w[e]);
                amax = fmaxf(amax, fabsf(w[e]));
                emax = fmaxf(emax, fabsf(w[e] - a));
                hi = fmaxf(hi, w[e]);
                lo = fminf(lo, w[e]);
            }
        x_sub[t >> 2] = v.x;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        }
        const int64_t j = t / kEnvG;
        if ((threadIdx.x & 3) == 0 && j < nblk) {
            mx0[j] = hi;
            mn0[j] = lo;
        }
    }
    unsigned ua = __float_as_uint(amax), ue = __float_as_uint(emax);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ua = max(ua, __shfl_xor_sync(0xffffffffu, ua, o));
        ue = max(ue, __shfl_xor_sync(0xffffffffu, ue, o));
    }
    const bool anybad = __any_sync(0xffffffffu, bad);
    if (lane_id() == 0) {
        if (anybad) atomicOr(flag, 1);
        if (ua) atomicMax(absmax, ua);
        if (ue) atomicMax(excursion, ue);
    }
}

cudaError_t launch_series_first(const float *x, int64_t n, int *flag, unsigned *absmax, unsigned *excursion,
                                float *x_sub, float *st, int64_t nblk, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(excursion, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const int64_t nb = (n + kBlockB - 1) / kBlockB;
    k_series_first<<<(unsigned)nb, kFirstThreads, 0, s>>>(x, n, flag, absmax, excursion, x_sub, st,
                                                          st + (size_t)kEnvLevels * nblk, nblk);
    return cudaGetLastError();
}

__global__ void k_fill(float *__restrict__ p, int64_t count, float v) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x)
        p[t] = v;
}

cudaError_t launch_fill(float *p, int64_t count, float v, int num_sms, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 8LL * num_sms) blocks = 8LL * num_sms;
    k_fill<<<(int)blocks, 256, 0, s>>>(p, count, v);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ FP32 pairs
__device__ __forceinline__ f2 ld2(const float *h, const float *l, int64_t t) { return {h[t], l[t]}; }

// ------------------------------------------------------------------ prefix
// One CTA per block b of kBlockB samples.  The anchor a_b = x[b*B]; every sum
// inside the block runs over d = x - a_b, so no sum grows with the series.
// Outputs, for t in block b:
//   P1[t] = sum_{bB <= u < t} d_u,  P2[t] = sum d_u^2   (exclusive prefix)
//   T1[b], T2[b] = block totals, A[b] = a_b,
//   ok[b] = 1 when every nonzero |d| in the block lies in [2^-40, 2^40], so
//   that no pair over- or underflows FP32 (else windows touching the block
//   take the two-pass FP64 path).
// Each prefix is stored as the pair hi = fl32(v), lo = fl32(v - hi)
// (|v - hi - lo| <= 2^-48 |v|), so the per-window arithmetic runs in FP32
// pairs.  All of it in units scaled by one power of two per series, 2^s with
// s such that the largest in-block excursion max|x - a_b| lies in [1, 2)
// (exact scaling; it keeps the pairs away from FP32 over- and underflow
// whatever the series' units).  Layout: pf = [P1h | P1l | P2h | P2l]
// (prefix_stride(n) floats each), bf = [T1h | T1l | T2h | T2l | A] (nb floats
// each, A scaled), scale[0] = 2^s.
//
// Arithmetic: FP32 with error-free transformations, no FP64 (this part issues
// it at 1/64 of the FP32 rate).  d is the exact pair TwoSum(x, -a); d^2 the
// exact sum of dh^2 (product and FMA residual), 2 dh dl (likewise) and dl^2;
// a running sum is three floats A + B + C, A and B updated by TwoSum, so only
// C rounds (second-order compensated summation, Klein 2006): a sum of B terms
// is exact to about B^2 2^-72 of its largest partial sum, well inside the
// pair that stores it.  A thread owns kPfPer consecutive samples: it sums
// them, the CTA scans the threads' sums (warp shuffles, then across warps),
// and the thread sums them again from its carry and stores every prefix.
// Bound by FP32 issue (~160 instructions per sample; 4 B read and 16 B
// written).  Measured per 1e7 samples: 0.10 ms, against 8.97 ms (9.9 ms per 1e8)
// with one thread per block and FP64 Neumaier sums -- a serial chain of 8192
// samples whatever the series' length.
__device__ __forceinline__ f3 f3_sum(f3 x, f3 y) {
    f3_add(x, y.a, y.b);
    x.c = __fadd_rn(x.c, y.c);
    return x;
}
__device__ __forceinline__ f3 f3_shfl_up(f3 v, int o) {
    return {__shfl_up_sync(0xffffffffu, v.a, o), __shfl_up_sync(0xffffffffu, v.b, o),
            __shfl_up_sync(0xffffffffu, v.c, o)};
}
// the pair that stores a sum: hi = fl32 of it, lo the rest
__device__ __forceinline__ f2 f3_pair(const f3 &t) {
    const exact2 p = two_sum_rn(t.a, t.b);
    const float l = __fadd_rn(p.e, t.c), hi = __fadd_rn(p.s, l);
    return {hi, __fsub_rn(l, __fsub_rn(hi, p.s))};
}

constexpr int kPfThreads = 512, kPfPer = kBlockB / kPfThreads, kPfWarps = kPfThreads / 32;
__global__ void __launch_bounds__(kPfThreads)
k_prefix(const float *__restrict__ x, int64_t n, float *__restrict__ pf, float *__restrict__ bf,
         int *__restrict__ ok, int64_t nb, int64_t stride, const unsigned *__restrict__ excursion,
         float *__restrict__ scale_out) {
    static_assert(kPfPer % 4 == 0 && kPfWarps <= 32, "whole float4s per thread, one scan across warps");
    __shared__ f3 w1[kPfWarps], w2[kPfWarps];
    const int64_t b = blockIdx.x, t0 = b * kBlockB + (int64_t)threadIdx.x * kPfPer;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const float mx = __uint_as_float(*excursion);
    // 2^s with mx * 2^s in [1, 2); 1 for a constant series
    const float sc = mx > 0.0f ? (float)ldexp(1.0, -ilogbf(mx)) : 1.0f;
    if (b == 0 && threadIdx.x == 0) scale_out[0] = sc;
    const float a = x[b * kBlockB];
    float xv[kPfPer];
#pragma unroll
    for (int q = 0; q < kPfPer / 4; ++q) {
        const float4 v = reinterpret_cast<const float4 *>(x + t0)[q];
        xv[4 * q] = v.x;
        xv[4 * q + 1] = v.y;
        xv[4 * q + 2] = v.z;
        xv[4 * q + 3] = v.w;
    }
    // d = x - a, scaled; samples past the series add nothing
    auto diff = [&](int e) {
        exact2 d = two_sum_rn(t0 + e < n ? xv[e] : a, -a);
        d.s = __fmul_rn(d.s, sc);
        d.e = __fmul_rn(d.e, sc);
        return d;
    };
    f3 s1{0.0f, 0.0f, 0.0f}, s2{0.0f, 0.0f, 0.0f};
    bool good = true;
#pragma unroll
    for (int e = 0; e < kPfPer; ++e) {
        const exact2 d = diff(e);
        const float ad = fabsf(d.s);
        good &= d.s == 0.0f || (ad >= 0x1p-40f && ad <= 0x1p40f);  // (NaN: not good)
        f3_add(s1, d.s, d.e);
        f3_add_sq(s2, d.s, d.e);
    }
    // inclusive scan of the threads' sums within the warp, then of the warps'
    f3 i1 = s1, i2 = s2;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const f3 u1 = f3_shfl_up(i1, o), u2 = f3_shfl_up(i2, o);
        if (lane >= o) {
            i1 = f3_sum(u1, i1);
            i2 = f3_sum(u2, i2);
        }
    }
    if (lane == 31) {
        w1[warp] = i1;
        w2[warp] = i2;
    }
    const bool all_good = __syncthreads_and(good);
    if (warp == 0) {
        f3 v1{0.0f, 0.0f, 0.0f}, v2{0.0f, 0.0f, 0.0f};
        if (lane < kPfWarps) {
            v1 = w1[lane];
            v2 = w2[lane];
        }
#pragma unroll
        for (int o = 1; o < kPfWarps; o <<= 1) {
            const f3 u1 = f3_shfl_up(v1, o), u2 = f3_shfl_up(v2, o);
            if (lane >= o) {
                v1 = f3_sum(u1, v1);
                v2 = f3_sum(u2, v2);
            }
        }
        if (lane < kPfWarps) {
            w1[lane] = v1;
            w2[lane] = v2;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const f2 p1 = f3_pair(w1[kPfWarps - 1]), p2 = f3_pair(w2[kPfWarps - 1]);
        bf[b] = p1.hi;
        bf[nb + b] = p1.lo;
        bf[2 * nb + b] = p2.hi;
        bf[3 * nb + b] = p2.lo;
        const float as = __fmul_rn(a, sc);
        bf[4 * nb + b] = as;
        // (the scaled anchor must be exact, so that scaling it back gives a)
        ok[b] = all_good && (double)as == (double)a * (double)sc && fabsf(as) < 1e30f ? 1 : 0;
    }
    // this thread's carry: the warps before, then the lanes before
    f3 c1 = f3_shfl_up(i1, 1), c2 = f3_shfl_up(i2, 1);
    if (lane == 0) c1 = c2 = f3{0.0f, 0.0f, 0.0f};
    if (warp > 0) {
        c1 = f3_sum(w1[warp - 1], c1);
        c2 = f3_sum(w2[warp - 1], c2);
    }
#pragma unroll
    for (int q = 0; q < kPfPer / 4; ++q) {
        f2 o1[4], o2[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            o1[e] = f3_pair(c1);
            o2[e] = f3_pair(c2);
            const exact2 d = diff(4 * q + e);
            f3_add(c1, d.s, d.e);
            f3_add_sq(c2, d.s, d.e);
        }
        // (the arrays hold whole blocks: prefix_stride)
        const int64_t t = t0 + 4 * q;
        *reinterpret_cast<float4 *>(pf + t) = make_float4(o1[0].hi, o1[1].hi, o1[2].hi, o1[3].hi);
        *reinterpret_cast<float4 *>(pf + stride + t) = make_float4(o1[0].lo, o1[1].lo, o1[2].lo, o1[3].lo);
        *reinterpret_cast<float4 *>(pf + 2 * stride + t) = make_float4(o2[0].hi, o2[1].hi, o2[2].hi, o2[3].hi);
        *reinterpret_cast<float4 *>(pf + 3 * stride + t) = make_float4(o2[0].lo, o2[1].lo, o2[2].lo, o2[3].lo);
    }
}

cudaError_t launch_prefix(const float *x, int64_t n, float *pf, float *bf, int *ok, const unsigned *excursion,
                          float *scale, cudaStream_t s) {
    const int64_t nb = (n + kBlockB - 1) / kBlockB;
    k_prefix<<<(unsigned)nb, kPfThreads, 0, s>>>(x, n, pf, bf, ok, nb, prefix_stride(n), excursion, scale);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ window stats
// Eq. 5 statistics of window i = [i, i+m) from the anchored sums.  A window
// spans at most two blocks (m <= kBlockB); the second block's sums are moved
// to the first anchor with the exact shift identities
//   sum(x - a0)   = sum(x - a1) + k (a1 - a0)
//   sum(x - a0)^2 = sum(x - a1)^2 + 2 (a1 - a0) sum(x - a1) + k (a1 - a0)^2,
// all in FP32 pairs (about 2^-47 relative per operation).  var = S2/m - (S1/m)^2.
// The window is evaluated two-pass from its samples instead when
//   * a block it touches is not ok (see k_prefix), or
//   * the subtraction cancelled, var <= 1e-6 * S2/m, or
//   * var is below the bound the sums' rounding implies.  With e1, e2 the bounds
//     of f2_diff, S1 is off by no more than 2^-48 e1, S2 by 2^-48 e2, and the
//     pair operations on them by less than 2^-48 12 S2 of m var; var then holds
//     2^-26 relative accuracy only if m*var >= 2^-22 (e2 + 12 S2 + 2|S1/m| e1).  (A
//     window over two blocks takes the totals M2 of its blocks' squares and
//     the shift terms instead: 3 M2 + 4|S1/m| sqrt(B M2).  That bound for
//     every window sent one in a hundred of a random walk's at m = 64 to the
//     two-pass evaluation.)
// Zero-variance rule: var <= 1e-24*max(1, mu^2) gives inv_sigma = 0 (the
// window normalises to all zeros).
//
// Bound by instruction issue (80 % of the slots at 284 instructions per
// window, 178 us per 2e7): so the pair operations keep only the steps that
// their result needs, a thread takes two adjacent windows at a time (its
// prefixes and results are float2s, two of them at i + m when m is odd), and
// a CTA's windows start in one block, whose anchor, flag and end it reads once.
// 2e7 windows of m = 512: 215 us with every step and one window per thread,
// 122 us now.
constexpr int kWsThreads = 256, kWsPer = 2, kWsIter = 4, kWsTile = kWsThreads * kWsPer * kWsIter;

struct StatsIn {
    const float *x, *pf, *bf;
    const int *ok;
    const float *scale;
    int64_t n, nb, stride;
    int m;
};

// p[i + S], p[i + S + 1], i even.  (One or two floats past the prefix arrays'
// end at most, inside their allocation; such a value belongs to no window.)
template <int S>
__device__ __forceinline__ float2 load_at(const float *p) {
    const float2 a = *reinterpret_cast<const float2 *>(p);
    return S == 0 ? a : make_float2(a.y, p[2]);
}
// The two-pass evaluation (near-constant windows, or blocks whose values the
// FP32 pairs cannot carry), by the window's thread: such windows come in runs,
// and sums in FP32 expansions (fp_sum.cuh) run at full rate where FP64 sums,
// or a warp per window with its FP64 reductions, are bound by the FP64 units
// (2e7 windows of m = 64, one in a hundred evaluated here: 0.65 and 1.1 ms).
__device__ __noinline__ float3 stats_two_pass(const float *__restrict__ x, int m) {
    double mu, var;
    mean_and_variance(x, m, 0, 1, [](double v) { return v; }, mu, var);
    float3 o;
    o.x = (float)mu;
    o.y = (float)(mu - (double)o.x);
    o.z = 0.0f;
    const double mm = mu * mu;
    if (!(var <= 1e-24 * (mm > 1.0 ? mm : 1.0))) {
        double y = (double)rsqrtf((float)var);
        y = y * fma(-0.5 * var * y, y, 1.5);
        o.z = (float)y;
    }
    return o;
}

template <int S>
__global__ void __launch_bounds__(kWsThreads, 4)
k_window_stats(StatsIn in, float *__restrict__ mu_hi, float *__restrict__ mu_lo, float *__restrict__ inv_sigma,
               float *__restrict__ smu_hi, float *__restrict__ sinv_sigma) {
    static_assert(kProxyStride % kWsPer == 0, "a window of the proxy scan is the first of a thread");
    static_assert(kBlockB % kWsTile == 0, "a CTA's windows start in one block");
    const int64_t N = in.n - in.m + 1, base = (int64_t)blockIdx.x * kWsTile, b0 = base / kBlockB;
    const int m = in.m;
    const float sc = in.scale[0], isc = 1.0f / sc;  // powers of two
    const float *t1h = in.bf, *t1l = in.bf + in.nb, *t2h = in.bf + 2 * in.nb, *t2l = in.bf + 3 * in.nb,
                *A = in.bf + 4 * in.nb;
    // 1/m as a pair: hi = fl(1/m), lo = (1 - hi*m)/m (the FMA residual is exact)
    const float ih = 1.0f / (float)m;
    const f2 inv_m = {ih, fmaf(-ih, (float)m, 1.0f) * ih};
    const float a0 = A[b0];
    const bool ok0 = in.ok[b0] != 0;
    // in samples from `base`: the block's end, the block's or the series' end
    const int end0 = (int)((b0 + 1) * kBlockB - base);
    const int tot0 = (int)((in.n < (b0 + 1) * kBlockB ? in.n : (b0 + 1) * kBlockB) - base);
    const int left = (int)(N - base < kWsTile ? N - base : kWsTile);
#pragma unroll 1
    for (int j = (int)threadIdx.x * kWsPer; j < left; j += kWsThreads * kWsPer) {
        const int64_t i0 = base + j;
        const float *p = in.pf + i0, *pe = p + (m - S);
        const float2 s1h = load_at<0>(p), s1l = load_at<0>(p + in.stride), s2h = load_at<0>(p + 2 * in.stride),
                     s2l = load_at<0>(p + 3 * in.stride);
        const float2 e1h = load_at<S>(pe), e1l = load_at<S>(pe + in.stride), e2h = load_at<S>(pe + 2 * in.stride),
                     e2l = load_at<S>(pe + 3 * in.stride);
        float mh[kWsPer], ml[kWsPer], is[kWsPer];
#pragma unroll
        for (int q = 0; q < kWsPer; ++q) {
            const int e = j + q + m;
            const f2 P1 = q ? f2{s1h.y, s1l.y} : f2{s1h.x, s1l.x}, P2 = q ? f2{s2h.y, s2l.y} : f2{s2h.x, s2l.x};
            f2 E1 = q ? f2{e1h.y, e1l.y} : f2{e1h.x, e1l.x}, E2 = q ? f2{e2h.y, e2l.y} : f2{e2h.x, e2l.x};
            f2 S1, S2;
            float err2, err1;  // errors of S2, S1 in units of 2^-48
            bool good = ok0;
            if (e <= end0) {
                if (e == tot0) {
                    E1 = ld2(t1h, t1l, b0);
                    E2 = ld2(t2h, t2l, b0);
                }
                S1 = f2_diff(E1, P1, err1);
                S2 = f2_diff(E2, P2, err2);
                err2 = fmaf(12.0f, S2.hi, err2);
            } else {
                const int64_t b1 = b0 + 1 < in.nb ? b0 + 1 : b0;  // (past N: unused)
                const int64_t end1 = (b1 + 1) * kBlockB;
                good = good && in.ok[b1] != 0;
                if (base + e == (end1 < in.n ? end1 : in.n)) {
                    E1 = ld2(t1h, t1l, b1);
                    E2 = ld2(t2h, t2l, b1);
                }
                const float k = (float)(e - end0);
                const f2 da = two_sum(A[b1], -a0);
                S1 = f2_add(f2_add(ld2(t1h, t1l, b0), f2_neg(P1)), f2_add(f2_mul_f(da, k), E1));
                const f2 da_e1 = f2_mul(da, E1);
                const f2 sh = f2_add(f2_add({2.0f * da_e1.hi, 2.0f * da_e1.lo}, f2_mul_f(f2_mul(da, da), k)), E2);
                S2 = f2_add(f2_add(ld2(t2h, t2l, b0), f2_neg(P2)), sh);
                const float M2 = t2h[b0] + t2h[b1] + 2.0f * fabsf(da.hi) * sqrtf((float)kBlockB * t2h[b1]) +
                                 k * da.hi * da.hi;
                err2 = 3.0f * M2;
                err1 = 2.0f * sqrtf((float)kBlockB * M2);
            }
            const f2 mr = f2_mul(S1, inv_m);
            // var = S2/m - mr^2 (the products unnormalised: their high parts
            // differ exactly, and the rest is summed at its own size)
            const float ph = __fmul_rn(S2.hi, inv_m.hi);
            const float pl = fmaf(S2.hi, inv_m.lo, fmaf(S2.lo, inv_m.hi, fmaf(S2.hi, inv_m.hi, -ph)));
            const float qh = __fmul_rn(mr.hi, mr.hi), ql = fmaf(2.0f * mr.hi, mr.lo, fmaf(mr.hi, mr.hi, -qh));
            f2 var2 = two_sum(ph, -qh);
            var2 = fast_two_sum(var2.hi, var2.lo + (pl - ql));
            f2 mu2 = two_sum(a0, mr.hi);
            mu2 = fast_two_sum(mu2.hi, mu2.lo + mr.lo);
            const float bound = 2.384185791015625e-07f *  // 2^-22
                                fmaf(2.0f * fabsf(mr.hi), err1, err2);
            mh[q] = mu2.hi * isc;
            ml[q] = mu2.lo * isc;
            is[q] = 0.0f;
            const float z = 1e-12f * fmaxf(sc, fabsf(mu2.hi));
            if (!good || var2.hi <= 1e-6f * ph || var2.hi * (float)m < bound) {
                if (j + q < left) {
                    const float3 o = stats_two_pass(in.x + i0 + q, m);
                    mh[q] = o.x;
                    ml[q] = o.y;
                    is[q] = o.z;
                }
            } else if (!(var2.hi <= z * z)) {
                // (the zero-variance rule in scaled units.)  1/sqrt(var): FP32
                // estimate refined by one Newton step whose residual 1 - var*y^2
                // is taken in pairs (the product's high part is near 1, so the
                // first difference is exact); then back to the series' units
                const float y = rsqrtf(var2.hi);
                const float yh = y * y, yl = fmaf(y, y, -yh);
                const float w = __fmul_rn(var2.hi, yh);
                const float we = fmaf(var2.hi, yh, -w) + fmaf(var2.hi, yl, var2.lo * yh);
                is[q] = fmaf(0.5f * y, __fsub_rn(__fsub_rn(1.0f, w), we), y) * sc;
            }
        }
        if (j + 1 < left) {
            *reinterpret_cast<float2 *>(mu_hi + i0) = make_float2(mh[0], mh[1]);
            *reinterpret_cast<float2 *>(mu_lo + i0) = make_float2(ml[0], ml[1]);
            *reinterpret_cast<float2 *>(inv_sigma + i0) = make_float2(is[0], is[1]);
        } else {
            mu_hi[i0] = mh[0];
            mu_lo[i0] = ml[0];
            inv_sigma[i0] = is[0];
        }
        // every kProxyStride-th window, for the proxy scan (the mean's high
        // part alone: the proxy only ranks proposals)
        if (j % kProxyStride == 0) {
            smu_hi[i0 / kProxyStride] = mh[0];
            sinv_sigma[i0 / kProxyStride] = is[0];
        }
    }
}

cudaError_t launch_window_stats(const float *x, int64_t n, int m, const float *pf, const float *bf,
                                const int *ok, const float *scale, float *mu_hi, float *mu_lo, float *inv_sigma,
                                float *smu_hi, float *sinv_sigma, cudaStream_t s) {
    const int64_t N = n - m + 1, nb = (n + kBlockB - 1) / kBlockB;
    const unsigned blocks = (unsigned)((N + kWsTile - 1) / kWsTile);
    const StatsIn in{x, pf, bf, ok, scale, n, nb, prefix_stride(n), m};
    if (m & 1)
        k_window_stats<1><<<blocks, kWsThreads, 0, s>>>(in, mu_hi, mu_lo, inv_sigma, smu_hi, sinv_sigma);
    else
        k_window_stats<0><<<blocks, kWsThreads, 0, s>>>(in, mu_hi, mu_lo, inv_sigma, smu_hi, sinv_sigma);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ envelope
// U[t] = max x[max(0,t-r) .. min(n-1,t+r)], L[t] = min (clipped to the
// series; samples outside [0, n) count as -inf / +inf, which never wins).
// A window of w = 2r+1 >= 7 samples is the end of a group of four, a run of
// whole groups and the start of a group.  A CTA makes kEnvTile outputs: per
// sample the max (min) to the end of its group and from the start of its
// group (in registers, a group per thread and step), per group the max (min)
// of the 2^P groups from it on by doubling in shared memory, where 2^P is the
// largest power that the fewest whole groups of a window hold, so two
// overlapping runs cover them.  An output is then four values, whatever r.
// Bound by the shared-memory reads of the outputs (32 B each): 82 us for 2e7
// samples at r = 100, against 217 us with the doubling over single samples.
constexpr int kEnvTile = 4096;
constexpr int kEnvThreads = 512;
constexpr int kEnvGrp = 4;
constexpr int kEnvRMin = 3;  // a window of seven or more samples holds a whole group
constexpr int kEnvEdge = kEnvTile + kEnvGrp;  // samples an output's window can start (end) at, whole groups

__global__ void __launch_bounds__(kEnvThreads)
k_envelope(const float *__restrict__ x, int64_t n, int r, int pad, int span, float *__restrict__ U,
           float *__restrict__ L) {
    extern __shared__ __align__(16) float sm[];
    const int len = kEnvTile + 2 * pad, ng = len / kEnvGrp;  // pad: r rounded up to whole groups
    float *sx = sm, *px = sx + kEnvEdge, *sn = px + kEnvEdge, *pn = sn + kEnvEdge, *gx = pn + kEnvEdge, *gn = gx + ng;
    const int ge0 = (pad + r) / kEnvGrp;  // the group the first output's window ends in
    const int64_t t0 = (int64_t)blockIdx.x * kEnvTile;
    const float inf = __int_as_float(0x7f800000);
    for (int g = threadIdx.x; g < ng; g += kEnvThreads) {
        const int64_t t = t0 - pad + (int64_t)g * kEnvGrp;
        float a[4], c[4];
        if (t >= 0 && t + kEnvGrp <= n) {
            const float4 v = *reinterpret_cast<const float4 *>(x + t);
            a[0] = c[0] = v.x;
            a[1] = c[1] = v.y;
            a[2] = c[2] = v.z;
            a[3] = c[3] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool in = t + q >= 0 && t + q < n;
                const float v = in ? x[t + q] : 0.0f;
                a[q] = in ? v : -inf;
                c[q] = in ? v : inf;
            }
        }
        float4 p, u;
        p.x = a[0];
        p.y = fmaxf(p.x, a[1]);
        p.z = fmaxf(p.y, a[2]);
        p.w = fmaxf(p.z, a[3]);
        u.w = a[3];
        u.z = fmaxf(u.w, a[2]);
        u.y = fmaxf(u.z, a[1]);
        u.x = p.w;
        const bool head = g < kEnvEdge / kEnvGrp, tail = g >= ge0 && g - ge0 < kEnvEdge / kEnvGrp;
        if (tail) reinterpret_cast<float4 *>(px)[g - ge0] = p;
        if (head) reinterpret_cast<float4 *>(sx)[g] = u;
        gx[g] = p.w;
        p.x = c[0];
        p.y = fminf(p.x, c[1]);
        p.z = fminf(p.y, c[2]);
        p.w = fminf(p.z, c[3]);
        u.w = c[3];
        u.z = fminf(u.w, c[2]);
        u.y = fminf(u.z, c[1]);
        u.x = p.w;
        if (tail) reinterpret_cast<float4 *>(pn)[g - ge0] = p;
        if (head) reinterpret_cast<float4 *>(sn)[g] = u;
        gn[g] = p.w;
    }
    __syncthreads();
    constexpr int kPer = (kEnvTile + 2 * kMMax) / kEnvGrp / kEnvThreads;
    static_assert(kPer * kEnvThreads * kEnvGrp >= kEnvTile + 2 * kMMax, "every group in one step of the doubling");
    for (int h = 1; h < span; h *= 2) {
        // (a run that would pass the last group is needed by no output)
        float a[kPer], c[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int g = q * kEnvThreads + (int)threadIdx.x;
            if (g < ng) {
                const int v = g + h < ng ? g + h : ng - 1;
                a[q] = fmaxf(gx[g], gx[v]);
                c[q] = fminf(gn[g], gn[v]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int g = q * kEnvThreads + (int)threadIdx.x;
            if (g < ng) {
                gx[g] = a[q];
                gn[g] = c[q];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < kEnvTile / kEnvThreads; ++q) {
        const int o = q * kEnvThreads + (int)threadIdx.x;
        if (t0 + o >= n) break;
        const int u = o + pad - r, e = u + 2 * r;        // the window's first and last sample
        const int f = (u + kEnvGrp - 1) / kEnvGrp, l = (e + 1) / kEnvGrp - span;  // the runs of whole groups
        const int ee = e - ge0 * kEnvGrp;
        U[t0 + o] = fmaxf(fmaxf(sx[u], px[ee]), fmaxf(gx[f], gx[l]));
        L[t0 + o] = fminf(fminf(sn[u], pn[ee]), fminf(gn[f], gn[l]));
    }
}

// Bands below kEnvRMin: the window's samples, from L1.
__global__ void __launch_bounds__(256)
k_envelope_small(const float *__restrict__ x, int64_t n, int r, float *__restrict__ U, float *__restrict__ L) {
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (t >= n) return;
    const int64_t a = t - r > 0 ? t - r : 0, b = t + r < n - 1 ? t + r : n - 1;
    float u = x[t], l = u;
    for (int64_t j = a; j <= b; ++j) {
        const float v = x[j];
        u = fmaxf(u, v);
        l = fminf(l, v);
    }
    U[t] = u;
    L[t] = l;
}

cudaError_t launch_envelope(const float *x, int64_t n, int r, float *U, float *L, cudaStream_t s) {
    if (r < kEnvRMin) {
        k_envelope_small<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, n, r, U, L);
        return cudaGetLastError();
    }
    const int pad = (r + kEnvGrp - 1) / kEnvGrp * kEnvGrp, len = kEnvTile + 2 * pad;
    const int fewest = (2 * r + 1 - (kEnvGrp - 1)) / kEnvGrp;  // whole groups in a window: this many or one more
    int span = 1;
    while (2 * span <= fewest) span *= 2;
    const int64_t blocks = (n + kEnvTile - 1) / kEnvTile;
    const size_t smem = (size_t)(4 * kEnvEdge + 2 * (len / kEnvGrp)) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_envelope, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    k_envelope<<<(unsigned)blocks, kEnvThreads, smem, s>>>(x, n, r, pad, span, U, L);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ block envelope
// Sparse table over blocks of kEnvG samples: level 0 holds each block's max
// (min; written by k_series_first), level k the max (min) of blocks
// [j, j + 2^k); entries whose range passes the last block are left unset and
// never read.  A CTA makes every level of kLvTile blocks from those blocks
// and the 2^(kEnvLevels-1) - 1 after them, doubling in shared memory: level 0
// is read twice and each level written once (one launch per level read the
// previous level from L2 twice and took 6.6 us each at 1e7 samples).
constexpr int kLvTile = 1024, kLvSpan = kLvTile + (1 << (kEnvLevels - 1)), kLvThreads = 512;
__global__ void __launch_bounds__(kLvThreads) k_env_levels(float *__restrict__ mx, float *__restrict__ mn,
                                                           int64_t nblk) {
    __shared__ float u[kLvSpan], l[kLvSpan];
    constexpr int kPer = (kLvSpan + kLvThreads - 1) / kLvThreads;
    const int64_t j0 = (int64_t)blockIdx.x * kLvTile;
    const float inf = __int_as_float(0x7f800000);
    for (int i = threadIdx.x; i < kLvSpan; i += kLvThreads) {
        const bool in = j0 + i < nblk;
        u[i] = in ? mx[j0 + i] : -inf;
        l[i] = in ? mn[j0 + i] : inf;
    }
    __syncthreads();
    for (int k = 1; k < kEnvLevels; ++k) {
        const int h = 1 << (k - 1);
        const int64_t last = nblk - (1ll << k);
        float a[kPer], c[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int i = q * kLvThreads + (int)threadIdx.x;
            // (past the span's end the run is not needed by any output)
            const int v = i + h < kLvSpan ? i + h : kLvSpan - 1;
            a[q] = i < kLvSpan ? fmaxf(u[i], u[v]) : 0.0f;
            c[q] = i < kLvSpan ? fminf(l[i], l[v]) : 0.0f;
        }
        __syncthreads();
        float *qm = mx + (size_t)k * nblk, *qn = mn + (size_t)k * nblk;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int i = q * kLvThreads + (int)threadIdx.x;
            if (i < kLvSpan) {
                u[i] = a[q];
                l[i] = c[q];
            }
            if (i < kLvTile && j0 + i <= last) {
                qm[j0 + i] = a[q];
                qn[j0 + i] = c[q];
            }
        }
        __syncthreads();
    }
}

cudaError_t launch_block_envelope(float *st, int64_t nblk, cudaStream_t s) {
    k_env_levels<<<(unsigned)((nblk + kLvTile - 1) / kLvTile), kLvThreads, 0, s>>>(
        st, st + (size_t)kEnvLevels * nblk, nblk);
    return cudaGetLastError();
}

}  // namespace dtws
