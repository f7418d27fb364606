// dtw_at64.cu -- extended-precision banded DTW at many given offsets of a
// handle's series: the double-float walk (dtw_band.cuh) arranged for the
// grid's rate.
#include "dtw_at.cuh"
#include "fp_sum.cuh"

namespace dtws {

namespace {

// The walk is bound by instruction issue.  In its general form a cell costs
// ~41 instructions, and with the register windows' moves, the half-rate
// selects and the cells past the band 84 issue slots per cell of the band
// (m = 1024, r = 102).  Here
//   * the minimum of three pairs is a three-input minimum of the high parts,
//     then one of the low parts, where a high part above the minimum lifts its
//     low part out of reach: 2 minima and 6 operations of the FMA pipe instead
//     of 6 comparisons and 4 selects, which issue at half rate;
//   * the square stays unnormalised (4 operations instead of 7): its parts are
//     added to the path's sum one after the other;
//   * odd cell counts, whose lanes load their own register windows (dtw_diag),
//     and a spare cell, so that the neighbour exchange may wrap;
//   * window values come raw from L1 and are normalised by the lane that takes
//     them, one per pair of steps (19 operations): staged copies of 8 bytes a
//     sample left 8 warps on an SM, which issued in 64 % of the cycles;
//   * the register windows move by copies (2 K per pair of steps): rotated in
//     place over K unrolled pairs, as dtw_diag's, the loop outgrew the
//     instruction cache (60 KB at K = 7: two thirds of the stalls).
// (Splitting the values on a common grid,
// so that a difference takes 2 operations instead of 11, was 1.3 times as fast
// again, but carries 2^-45 of the largest value instead of 2^-48 of each: ten
// times the error on a near match.)  Measured, 4,096 windows: m = 1024,
// r = 102 1.94 -> 1.38 ms, m = 2048, r = 204 9.0 -> 5.2, m = 512, r = 51 0.59 ->
// 0.45; the errors against 64 bits are the general walk's (mean 1.9e-14 at
// m = 1024).
// one CTA per SM, as many threads as the registers allow without a spill (at
// seven cells 16 warps with spills were no faster than 12, and slower alone)
__host__ __device__ constexpr int r64_threads(int K) { return K <= 5 ? 512 : K <= 7 ? 384 : 256; }

// A window's normalisation: its mean in three parts (it may be many sigma, and
// its error is every value's), 1/sigma in two.  Samples and mean are taken
// times the power of two f that brings 1/sigma into [1, 2), whatever the
// series' units: at sigma = 1e36 the low part of 1/sigma itself is subnormal
// (2e-9 of it), and the difference of two samples of either sign overflows.
struct R64Norm {
    float f, m1, m2, m3, ih, il;
};
// (The exponents are added as integers: FP64 issues at 1/64 of FP32's rate here,
// and ldexp and ilogb took 1 % of a walk.  A mean of FP32 samples is zero or a
// normal FP64 value, and so is it times 2^-126 .. 2^40.)
__device__ __forceinline__ double times_pow2(double v, int e) {
    return v == 0.0 ? v : __hiloint2double(__double2hiint(v) + e * (1 << 20), __double2loint(v));
}
__device__ __forceinline__ R64Norm r64_scaled(double mu, double inv) {
    // inv's exponent; 0 for no sigma, where every value is 0 (2^-126 is the least
    // that is normal in FP32: 1/sigma >= 2^-128 is then 2^-2 or more)
    const int e = inv > 0.0 ? max((__double2hiint(inv) >> 20) - 1023, -126) : 0;
    const double sm = times_pow2(mu, e);
    const dfloat m = df_from(sm), v = df_from(times_pow2(inv, -e));
    return R64Norm{__int_as_float((e + 127) << 23), m.hi, m.lo, (float)(sm - (double)m.hi - (double)m.lo), v.hi, v.lo};
}
__device__ __forceinline__ dfloat r64_norm(const R64Norm &n, float x) {
    const dfloat s = df_two_sum(__fmul_rn(x, n.f), -n.m1), u = df_two_sum(s.hi, -n.m2);
    const dfloat d = df_fast_two_sum(u.hi, __fadd_rn(s.lo, u.lo) - n.m3);
    const float p = __fmul_rn(d.hi, n.ih);
    return df_fast_two_sum(p, fmaf(d.hi, n.il, fmaf(d.lo, n.ih, fmaf(d.hi, n.ih, -p))));
}

// One anti-diagonal (as diag_step with SPARE).
template <int L, int K, int ODD>
__device__ __forceinline__ void r64_step(const dfloat (&qv)[K], const dfloat (&cv)[K], dfloat (&p1)[K], dfloat (&p2)[K],
                                         const float (&pen)[K], int lane, unsigned gmask) {
    const dfloat nb = df_shfl(gmask, ODD ? p1[0] : p1[K - 1], ODD ? ((lane + 1) & (L - 1)) : ((lane - 1) & (L - 1)), L);
    dfloat cur[K];
#pragma unroll
    for (int t = 0; t < K; ++t) {
        const dfloat left = ODD ? p1[t] : (t == 0 ? nb : p1[t > 0 ? t - 1 : 0]);
        const dfloat up = ODD ? (t == K - 1 ? nb : p1[t < K - 1 ? t + 1 : 0]) : p1[t];
        const dfloat d = df_sub(qv[t], cv[t]);
        float p = __fmul_rn(d.hi, d.hi);
        const float e = fmaf(d.hi + d.hi, d.lo, fmaf(d.hi, d.hi, -p));
        // the least of the three, high parts first (they are finite, and low
        // parts are at most 2^-24 of them)
        const float bh = min3f(left.hi, up.hi, p2[t].hi);
        const float bl = min3f(fmaf(__fsub_rn(left.hi, bh), 0x1p60f, left.lo),
                               fmaf(__fsub_rn(up.hi, bh), 0x1p60f, up.lo),
                               fmaf(__fsub_rn(p2[t].hi, bh), 0x1p60f, p2[t].lo));
        if (ODD) p = __fadd_rn(p, pen[t]);
        const dfloat s = df_two_sum(bh, p);
        cur[t] = df_fast_two_sum(s.hi, __fadd_rn(__fadd_rn(s.lo, e), bl));
    }
#pragma unroll
    for (int t = 0; t < K; ++t) {
        p2[t] = p1[t];
        p1[t] = cur[t];
    }
}

// The walk of one window by a group of L lanes (dtw_diag's, without abandon).
// qs: the query's double-floats, padded by diag_pad; xw: the window's samples.
template <int L, int K>
__device__ __forceinline__ double r64_walk(const dfloat *__restrict__ qs, const float *__restrict__ xw, int m, int r,
                                           const R64Norm &norm, unsigned gmask, int lane) {
    static_assert(K & 1, "every lane loads its own values");
    const dfloat INF = dfloat{1e30f, 0.0f}, out = dfloat{-1e15f, 0.0f};
    const int p0 = (r - (r & 1)) >> 1, last = 2 * m - 2;
    dfloat p1[K], p2[K], qv[K], cv[K];
    float pen[K];
#pragma unroll
    for (int t = 0; t < K; ++t) {
        p1[t] = INF;
        p2[t] = (lane * K + t == p0) ? dfloat{0.0f, 0.0f} : INF;
        pen[t] = lane * K + t >= r ? 1e30f : 0.0f;
    }
    const dfloat *qp = qs - lane * K;
    const int c0 = lane * K;
    // sample c0 + j of the window (any one when there is none), its value
    auto raw = [&](int j) { return __ldg(xw + min(max(c0 + j, 0), m - 1)); };
    auto value = [&](float x, int j) {
        const dfloat v = r64_norm(norm, x);
        return (unsigned)(c0 + j) < (unsigned)m ? v : out;
    };
    int a = -(r & 1), bi = (a + r) >> 1, bj = (a - r) >> 1;
#pragma unroll
    for (int t = 0; t < K; ++t) {
        qv[t] = qp[bi - t];
        cv[t] = value(raw(bj + t), bj + t);
    }
    if (r & 1) {
        // the base cell lies one anti-diagonal before a = -1, whose cells are
        // all outside the matrix
#pragma unroll
        for (int t = 0; t < K; ++t) {
            p1[t] = p2[t];
            p2[t] = INF;
        }
    }
#pragma unroll 1
    for (;; a += 2, ++bi, ++bj) {
        const float x = raw(bj + K);
        const dfloat q = qp[bi + 1];
        r64_step<L, K, 0>(qv, cv, p1, p2, pen, lane, gmask);
        if (a == last) break;
#pragma unroll
        for (int t = 0; t < K - 1; ++t) cv[t] = cv[t + 1];
        cv[K - 1] = value(x, bj + K);
        r64_step<L, K, 1>(qv, cv, p1, p2, pen, lane, gmask);
        if (a + 1 == last) break;
#pragma unroll
        for (int t = K - 1; t > 0; --t) qv[t] = qv[t - 1];
        qv[0] = q;
    }
    const int pe = (r - ((last + r) & 1)) >> 1;
    dfloat res = INF;
#pragma unroll
    for (int t = 0; t < K; ++t)
        if (lane * K + t == pe) res = p1[t];
    res = df_shfl(gmask, res, pe / K, L);
    return (double)res.hi + (double)res.lo;
}

template <int L, int K>
__global__ void __launch_bounds__(r64_threads(K), 1)
k_dtw64_many(QueryBufs b, QueryArgs a, const int64_t *__restrict__ offsets, int64_t count, double *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smraw[];
    if (!b.st->valid) return;
    constexpr int kThr = r64_threads(K), kPer = 32 / L;
    const int m = a.m, r = a.r, pad = diag_pad(r, L, K);
    dfloat *qs = (dfloat *)smraw + pad;
    for (int t = threadIdx.x; t < m; t += kThr) qs[t] = df_from(b.qh64[t]);
    for (int t = threadIdx.x; t < 2 * pad; t += kThr) qs[t < pad ? t - pad : m + t - pad] = dfloat{1e15f, 0.0f};
    __syncthreads();
    const int ln = lane_id(), g = ln / L, lane = ln % L;
    // few windows go to one warp of each scheduler, then to its other groups,
    // then to the next four warps
    const int warp = (int)(threadIdx.x >> 5), gid = warp / 4 * 4 * kPer + g * 4 + warp % 4;
    const unsigned gmask = (L == 32) ? 0xffffffffu : (((1u << L) - 1u) << (g * L));
    auto gsum = [&](double v) {
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gmask, v, o, L);
        return v;
    };
    // (neighbouring windows on different SMs: few windows still use them all)
    for (int64_t c = blockIdx.x + (int64_t)gid * gridDim.x; c < count; c += (int64_t)(kThr / L) * gridDim.x) {
        const int64_t o = offsets[c];
        if (o < 0 || o >= a.N) {
            if (lane == 0) out[c] = __longlong_as_double(0x7ff8000000000000ll);
            continue;
        }
        const float *xw = b.x + o;
        double mu, var;
        mean_and_variance(xw, m, lane, L, gsum, mu, var);
        const double inv = var <= 1e-24 * (mu * mu > 1.0 ? mu * mu : 1.0) ? 0.0 : 1.0 / sqrt(var);
        const double d = r64_walk<L, K>(qs, xw, m, r, r64_scaled(mu, inv), gmask, lane);
        if (lane == 0) out[c] = d;
    }
}

// Shapes: X(L, K).
#define DTWS_R64_SHAPES(X)                                                                                 \
    X(8, 3) X(8, 5) X(8, 7) X(8, 9) X(8, 11) X(8, 13) X(16, 3) X(16, 5) X(16, 7) X(16, 9) X(16, 11) X(16, 13) \
    X(32, 3) X(32, 5) X(32, 7) X(32, 9) X(32, 11) X(32, 13)
struct R64Plan {
    int L, K;
    size_t smem;
};
// Scheduler cycles of a warp's step and of a step that waits for itself alone,
// fitted to a sweep of every shape at 7 sizes (m = 128..4096, r = 12..409) and
// 5 counts (400..20,000): within 10 %.
inline double r64_issue(int L, int K) { return 45.0 * K + (L == 32 ? 35.0 : L == 16 ? 50.0 : 75.0); }
inline double r64_alone(int K) { return 70.0 + 51.0 * K; }
// Time per step of all windows when an SM has per_sm of them, `groups` at a
// time, `per` to a warp.
inline double r64_time(int64_t per_sm, int64_t groups, int per, double issue, double alone) {
    const int64_t rounds = (per_sm + groups - 1) / groups, some = rounds > 1 ? groups : per_sm;
    const double busy = (double)((some + 4 * per - 1) / (4 * per)) * issue, step = busy > alone ? busy : alone;
    return (rounds > 4 ? (double)per_sm / groups : (double)rounds) * step;
}
// The shape with the least time among those with L K >= r + 2.  False where
// the general walks are faster (dtw64_dispatch: one warp of K = 1..4 cells per
// lane up to r = 127, 120 cycles a step and 300 alone at K = 2) or the band has
// more than 414 cells: theirs are bands just below a power of two, which leave
// them no idle lane, of queries short enough that eight windows' copies and
// more fit an SM.  E.g. m = 1024, r = 60: 20,000 windows 4.25 ms there, 4.46 on
// (8, 9); 4,096 1.12 and 1.02; r = 102 7.83 and 6.17, 1.95 and 1.38.
bool r64_plan(int m, int r, int64_t count, int num_sms, R64Plan *best) {
    const int64_t per_sm = (count + num_sms - 1) / num_sms;
    const size_t copy = (size_t)(m + 2 * diag_pad(r, 32, 1)) * sizeof(dfloat), room = (size_t)200 * 1024;
    if (r < 16 && copy * 9 <= room) return false;
    double best_score = 1e300;
    if (r < 128) {
        const int K = r / 32 + 1;
        const int64_t groups = copy * 9 <= room ? 8 : (int64_t)(room / copy) - 1;
        if (groups > 0) {
            const int64_t ctas = (int64_t)((size_t)224 * 1024 / (copy * (size_t)(1 + groups)));
            best_score = r64_time(per_sm, groups * (ctas < 4 ? ctas : 4), 1, 50.0 * K + 20.0, 60.0 + 118.0 * K);
        }
    }
    bool found = false;
#define DTWS_R64_TRY(LL, KK)                                                                           \
    if (LL * KK >= r + 2) {                                                                            \
        const double score = r64_time(per_sm, r64_threads(KK) / LL, 32 / LL, r64_issue(LL, KK), r64_alone(KK)); \
        if (score < best_score) {                                                                      \
            found = true;                                                                              \
            best_score = score;                                                                        \
            *best = R64Plan{LL, KK, (size_t)(m + 2 * diag_pad(r, LL, KK)) * sizeof(dfloat)};           \
        }                                                                                              \
    }
    DTWS_R64_SHAPES(DTWS_R64_TRY)
#undef DTWS_R64_TRY
    return found;
}

template <int L, int K>
cudaError_t r64_launch(const QueryBufs &b, const QueryArgs &a, const int64_t *offsets, int64_t count, double *out,
                       const R64Plan &p, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_dtw64_many<L, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e != cudaSuccess) return e;
    k_dtw64_many<L, K><<<(unsigned)(count < b.num_sms ? count : b.num_sms), r64_threads(K), p.smem, s>>>(
        b, a, offsets, count, out);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dtw_at_f64_many(const QueryBufs &b, const QueryArgs &a, const int64_t *offsets, int64_t count,
                                   double *out, cudaStream_t s) {
    R64Plan p;
    // (raw values keep the walks of dtw64_dispatch)
    if (a.raw || count < 1 || !r64_plan(a.m, a.r, count, b.num_sms, &p)) return cudaErrorNotSupported;
#define DTWS_CASE(LL, KK) \
    if (p.L == LL && p.K == KK) return r64_launch<LL, KK>(b, a, offsets, count, out, p, s);
    DTWS_R64_SHAPES(DTWS_CASE)
#undef DTWS_CASE
    return cudaErrorInvalidValue;
}

}  // namespace dtws
