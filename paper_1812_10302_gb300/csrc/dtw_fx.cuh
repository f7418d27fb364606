// dtw_fx.cuh -- the extended-precision banded DTW of one window as fast as one
// CTA can walk it: 64-bit fixed-point path sums, costs formed by other warps.
#pragma once

#include "dtw_band.cuh"

namespace dtws {

// One window's re-score is pure latency: 2m - 1 dependent anti-diagonals.  In
// double-float (dtw_diag_df) a step costs ~41 instructions per cell, most of
// them the cell's cost, and one warp issued them all: 262 cycles per step at
// r = 51.  Here the CTA splits the work.  Eleven producer warps form the costs
// (q_hat_i - c_j)^2 of the coming anti-diagonals in double-float, as before,
// turn each into a 64-bit integer and leave it in a shared-memory ring; one
// consumer warp walks: per cell two integer minima and one addition (10
// instructions), per step one neighbour exchange by shuffle.  The two
// halves meet at a named barrier every kFxSteps anti-diagonals.
//
// The fixed point: with an upper bound U of the DTW (the caller's, or the
// diagonal path's cost) no partial sum above U lies on the best path.
// Costs are scaled by 2^s with U 2^s in (2^56, 2^58] and every cost at or
// above 2^59 saturates (cells outside the band or the matrix too).  Sums are
// then exact: the only rounding is each cost's, half a unit of 2^-s.  When the
// result comes out below kFxRedo units (a DTW far below the bound) the walk is repeated on the scale of that result, so a result
// always has at least 51 bits above its unit: with n rounded costs on the
// path its error is ~0.3 sqrt(n) 2^-51 relative, below the double-float walk's
// (measured against 64 bits over m = 32..2048: 1e-15 on average, against
// 2e-14).  Windows walked
// with the same bound (or with the diagonal's) score identically when their
// values are identical.
//
// Measured, dtws_dtw_at_f64 of one window, whole call: 105 us at m = 512,
// r = 51 (164 us before), 210 us at m = 1024, r = 102 (412 us); bound by the
// consumer's ALU issue (25 cycles per cell of a lane) past two cells per lane.
constexpr int kFxThreads = 384, kFxWarps = kFxThreads / 32, kFxSteps = 16, kFxUnit = 8;
// a saturated cost; the value saturated sums are set back to every kFxUnit
// steps (kFxInf + kFxUnit * kFxCost < 2^64, so no sum wraps in between)
constexpr unsigned long long kFxCost = 1ull << 60, kFxInf = 1ull << 61, kFxRedo = 1ull << 51;

// Cells per lane: 32 K >= r + 2, so the last cell of every anti-diagonal lies
// past the band and is always saturated; the neighbour exchange may then wrap
// around the warp without a special case.
__host__ __device__ inline int fx_cells(int r) {
    const int need = (r + 2 + 31) / 32;
    return need <= 4 ? need : need <= 6 ? 6 : 8;
}
constexpr int kFxRMax = 254;  // 32 * 8 - 2
__host__ __device__ constexpr size_t fx_ring_bytes(int K) {
    return (size_t)2 * kFxSteps * ((K + 1) / 2) * 32 * 16;
}
// Padding on each side of the query's and the window's double-floats: the
// producers' positions run to r/2 + 32 K + kFxSteps past either end.
__host__ __device__ inline int fx_pad(int r, int K) { return ((r >> 1) + 32 * K + kFxSteps + 4) & ~1; }
__host__ __device__ inline size_t fx_span(int m, int r, int K) { return (size_t)((m + 2 * fx_pad(r, K) + 1) & ~1); }
// shared memory of one window: the ring, the query's and the window's padded double-floats
__host__ __device__ inline size_t fx_bytes(int m, int r, int K) { return fx_ring_bytes(K) + fx_span(m, r, K) * 16; }
// whether a search re-scores with this walk (the pre-score needs its FP32
// walk's padded copies beside it): one rule for the pre-score and the final
// stage, so that equal windows are compared on equal terms
__host__ __device__ inline bool fx_used(int m, int r) {
    if (r > kFxRMax) return false;
    const int K = fx_cells(r);
    return fx_bytes(m, r, K) + (size_t)((m + 2 * diag_pad(r, 32, K) + 3) & ~3) * 8 <= (size_t)216 * 1024;
}

struct FxShared {
    float red[kFxWarps];
    unsigned long long res;
    double mu, inv;
};

__device__ __forceinline__ unsigned long long fx_min(unsigned long long x, unsigned long long y) {
    return x < y ? x : y;
}

// hi + lo in [0, 2^61), |lo| < 2^39, rounded to an integer by FP32 additions:
// adding 1.5 * 2^(23+u) to a float below 2^(22+u) leaves its multiple of 2^u in
// the low bits.  Three limbs (2^40, 2^17, 1) of hi and two of lo; every step is
// exact but the last.  The limbs' constant bits are taken off in one go (they
// start the sum).  (The conversion instruction to 64-bit integers runs at
// 1/64 rate on this part: with it the producers took 35 cycles of the SM per
// 32 cells.)
__device__ __forceinline__ unsigned long long fx_round(float hi, float lo) {
    constexpr float M2 = 0x1.8p63f, M1 = 0x1.8p40f, M0 = 0x1.8p23f;
    constexpr unsigned B2 = 0x5f400000u, B1 = 0x53c00000u, B0 = 0x4b400000u;  // their bit patterns
    constexpr unsigned long long kBias =
        ((unsigned long long)B2 << 40) + ((unsigned long long)(B1 + B1) << 17) + B0;
    const float a2 = hi + M2, r2 = hi - (a2 - M2);
    const float a1 = r2 + M1, r1 = r2 - (a1 - M1);
    const float b1 = lo + M1, q1 = lo - (b1 - M1);
    const float a0 = (r1 + q1) + M0;
    const unsigned s1 = __float_as_uint(a1) + __float_as_uint(b1);
    unsigned long long w = ((unsigned long long)__float_as_uint(a2) << 40) - kBias;
    w += (unsigned long long)s1 * (1u << 17);
    return w + __float_as_uint(a0);
}

// Costs of the virtual steps [v0, v0 + kFxUnit) (v0 even) for the cells
// p = blk * 32 + lane.  Virtual step v is anti-diagonal a = v - (r & 1), so
// that even v are even steps (a + r even); v = 0 with r odd is a = -1, which
// holds no cell.  Along a pair of steps the cell's row stays and its column
// grows by one, from pair to pair both grow by one, so a pair loads one query
// and one window value.  qd, cd are padded by fx_pad with poison (+1e15,
// -1e15): a cell outside [0, m)^2 comes out far above 2^59, as do sums that
// overflow, and everything not below 2^59 becomes kFxCost.  dst: the steps'
// ring slots.
template <int K>
__device__ __forceinline__ void fx_produce(const dfloat *qd, const dfloat *cd, int r, float f, int v0, int blk,
                                           unsigned long long *dst, int lane) {
    constexpr int kStep = ((K + 1) / 2) * 64;  // words of a step
    const int p = blk * 32 + lane, a = v0 - (r & 1);
    const dfloat *qp = qd + (((a + r) >> 1) - p), *cp = cd + (((a - r) >> 1) + p);
    const int pl = p / K, pt = p - pl * K;
    unsigned long long *o = dst + ((pt >> 1) * 32 + pl) * 2 + (pt & 1);
    const bool in0 = p <= r, in1 = p < r;  // cells of an even, of an odd step
    dfloat c = cp[0];
#pragma unroll
    for (int s = 0; s < kFxUnit; s += 2) {
        const dfloat q = qp[s / 2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (e) c = cp[s / 2 + 1];
            const dfloat d = df_sub(q, c);
            const float h = d.hi * f, l = d.lo * f;  // f is a power of two
            const float sq = __fmul_rn(h, h);
            const float er = fmaf(h + h, l, fmaf(h, h, -sq));
            const bool fine = (e ? in1 : in0) && sq < 0x1p59f;
            const unsigned long long w = fx_round(sq, er);
            o[(s + e) * kStep] = fine ? w : kFxCost;
        }
    }
}

// One anti-diagonal of the walk: cell t of the lane (as diag_step).
template <int K, int ODD>
__device__ __forceinline__ void fx_step(const unsigned long long *buf, unsigned long long (&p1)[K],
                                        unsigned long long (&p2)[K], int lane) {
    unsigned long long cost[((K + 1) / 2) * 2];
#pragma unroll
    for (int t = 0; t < (K + 1) / 2; ++t) {
        const ulonglong2 c = reinterpret_cast<const ulonglong2 *>(buf)[t * 32 + lane];
        cost[2 * t] = c.x;
        cost[2 * t + 1] = c.y;
    }
    const unsigned long long nb =
        __shfl_sync(0xffffffffu, ODD ? p1[0] : p1[K - 1], ODD ? ((lane + 1) & 31) : ((lane - 1) & 31));
    unsigned long long cur[K];
#pragma unroll
    for (int t = 0; t < K; ++t) {
        const unsigned long long left = ODD ? p1[t] : (t == 0 ? nb : p1[t > 0 ? t - 1 : 0]);
        const unsigned long long up = ODD ? (t == K - 1 ? nb : p1[t < K - 1 ? t + 1 : 0]) : p1[t];
        // (the neighbour lane's value last: only one minimum waits for it)
        const unsigned long long best = ODD ? fx_min(up, fx_min(left, p2[t])) : fx_min(left, fx_min(up, p2[t]));
        cur[t] = best + cost[t];
    }
#pragma unroll
    for (int t = 0; t < K; ++t) {
        p2[t] = p1[t];
        p1[t] = cur[t];
    }
}

// Saturated sums back to kFxInf (the high word decides; the low one may stay).
template <int K>
__device__ __forceinline__ void fx_clamp(unsigned long long (&v)[K]) {
#pragma unroll
    for (int t = 0; t < K; ++t) {
        const unsigned hi = min((unsigned)(v[t] >> 32), (unsigned)(kFxInf >> 32));
        v[t] = ((unsigned long long)hi << 32) | (unsigned)v[t];
    }
}

// The walk by the kFxThreads threads t = 0.. of a group that owns named
// barrier `bar`.  qd, cd: element 0 of q_hat and of the normalised window as
// double-floats, padded by fx_pad(r, K) elements of +1e15 and -1e15 on both
// sides; bound: an upper bound of the DTW, 0 for the diagonal path's cost;
// ring: fx_ring_bytes(K), 16-byte aligned.  Every thread returns
// the distance.
template <int K>
__device__ double dtw_fx(const dfloat *__restrict__ qd, const dfloat *__restrict__ cd, int m, int r, float bound,
                         int t, FxShared &sh, unsigned long long *ring, int bar) {
    const int lane = t & 31, warp = t >> 5;
    constexpr int kStep = ((K + 1) / 2) * 64;  // words of a step
    // the diagonal path's cost, an upper bound of the DTW (the same sum in every thread)
    auto euclid = [&]() {
        float ed = 0.0f;
        for (int j = t; j < m; j += kFxThreads) {
            const float d = df_sub(qd[j], cd[j]).hi;
            ed = fmaf(d, d, ed);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ed += __shfl_xor_sync(0xffffffffu, ed, o);
        if (lane == 0) sh.red[warp] = ed;
        group_bar(bar, kFxThreads);
        ed = 0.0f;
#pragma unroll
        for (int w = 0; w < kFxWarps; ++w) ed += sh.red[w];
        group_bar(bar, kFxThreads);  // (sh.red is read before it is written again)
        return ed;
    };
    auto scale_of = [](float bound) { return (58 - (ilogbf(bound * 1.001f) + 1)) >> 1; };
    if (!(bound > 0.0f && bound < 1e30f)) bound = euclid();
    if (!(bound > 0.0f)) return 0.0;  // (the Euclidean distance is 0)
    int h = scale_of(bound);          // the scale is 2^(2h)
    const int V = 2 * m - 1 + (r & 1), chunks = (V + kFxSteps - 1) / kFxSteps;
    const int p0 = (r - (r & 1)) >> 1, last = 2 * m - 2, pe = (r - ((last + r) & 1)) >> 1;
    for (int pass = 0;; ++pass) {
        const float f = ldexpf(1.0f, h);
        // a chunk's units: kFxUnit steps of one block of 32 cells each
        auto produce = [&](int c, int w, int nw) {
            unsigned long long *buf = ring + (size_t)(c & 1) * kFxSteps * kStep;
            for (int u = w; u < K * (kFxSteps / kFxUnit); u += nw) {
                const int blk = u % K, s0 = u / K * kFxUnit;
                fx_produce<K>(qd, cd, r, f, c * kFxSteps + s0, blk, buf + s0 * kStep, lane);
            }
        };
        produce(0, warp, kFxWarps);
        group_bar(bar, kFxThreads);
        unsigned long long p1[K], p2[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
            // the base cell lies on anti-diagonal -2: two steps before v = 0
            // when r is even, one before when r is odd
            const unsigned long long base = lane * K + u == p0 ? 0ull : kFxInf;
            p1[u] = (r & 1) ? base : kFxInf;
            p2[u] = (r & 1) ? kFxInf : base;
        }
        for (int c = 0; c < chunks; ++c) {
            const unsigned long long *buf = ring + (size_t)(c & 1) * kFxSteps * kStep;
            if (warp == 0) {
                const int steps = V - c * kFxSteps < kFxSteps ? V - c * kFxSteps : kFxSteps;
                if (steps == kFxSteps) {
#pragma unroll 1
                    for (int s0 = 0; s0 < kFxSteps; s0 += kFxUnit) {
#pragma unroll
                        for (int s = s0; s < s0 + kFxUnit; s += 2) {
                            fx_step<K, 0>(buf + s * kStep, p1, p2, lane);
                            fx_step<K, 1>(buf + (s + 1) * kStep, p1, p2, lane);
                        }
                        fx_clamp<K>(p1);
                        fx_clamp<K>(p2);
                    }
                } else {
                    for (int s = 0; s < steps; s += 2) {
                        fx_step<K, 0>(buf + s * kStep, p1, p2, lane);
                        if (s + 1 < steps) fx_step<K, 1>(buf + (s + 1) * kStep, p1, p2, lane);
                        if ((s + 2) % kFxUnit == 0) {
                            fx_clamp<K>(p1);
                            fx_clamp<K>(p2);
                        }
                    }
                }
            } else if (c + 1 < chunks) {
                produce(c + 1, warp - 1, kFxWarps - 1);
            }
            group_bar(bar, kFxThreads);
        }
        if (warp == 0) {
#pragma unroll
            for (int u = 0; u < K; ++u)
                if (lane * K + u == pe) sh.res = p1[u];
        }
        group_bar(bar, kFxThreads);
        const unsigned long long res = sh.res;
        group_bar(bar, kFxThreads);  // (sh.res is read before it is written again)
        if (res > (1ull << 59)) {  // `bound` did not hold: the Euclidean distance does
            bound = euclid();
            h = scale_of(bound);
            continue;
        }
        if (res >= kFxRedo || pass >= 3) return ldexp((double)res, -2 * h);
        // a DTW far below the bound: again on its own scale (its
        // V roundings allowed for), which puts it below 2^57; never past what
        // FP32 scales by (2^(2 * 120))
        const int up = (56 - (63 - __clzll((long long)(res + V)))) >> 1;
        if (h + up > 120) return ldexp((double)res, -2 * h);
        h += up;
    }
}

__device__ __forceinline__ void fill_pads_fx(dfloat *base, int m, int pad, dfloat v, int t) {
    for (int u = t; u < 2 * pad; u += kFxThreads) base[u < pad ? u : m + u] = v;
}

// The padded query and window copies behind the ring, their pads poisoned and
// the query filled, by the group's threads (the caller's next barrier, in
// fx_window, makes them visible).
template <int K>
__device__ __forceinline__ void fx_setup(unsigned char *sm, const double *__restrict__ qh64, int m, int r, int t,
                                         dfloat **qd, dfloat **cd) {
    const int pad = fx_pad(r, K);
    dfloat *q = (dfloat *)(sm + fx_ring_bytes(K)), *c = q + fx_span(m, r, K);
    fill_pads_fx(q, m, pad, dfloat{1e15f, 0.0f}, t);
    fill_pads_fx(c, m, pad, dfloat{-1e15f, 0.0f}, t);
    for (int j = t; j < m; j += kFxThreads) q[pad + j] = df_from(qh64[j]);
    *qd = q + pad;
    *cd = c + pad;
}

// Two-pass FP64 statistics (Eq. 5) of the window xw by the group's first warp
// into sh.mu, sh.inv (0 under the zero-variance rule; 0 and 1 for raw
// values), then its normalised values as double-floats.  All kFxThreads
// threads of the group call it; they have met at the barrier on return.
__device__ __forceinline__ void fx_window(const float *__restrict__ xw, int m, bool raw, dfloat *cd, FxShared &sh,
                                          int t, int bar) {
    const int lane = t & 31;
    if (t < 32) {
        double s = 0.0;
        for (int j = lane; j < m; j += 32) s += (double)xw[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const double mu = s / (double)m;
        double v = 0.0;
        for (int j = lane; j < m; j += 32) {
            const double d = (double)xw[j] - mu;
            v = fma(d, d, v);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            const double var = v / (double)m, mm = mu * mu;
            sh.mu = raw ? 0.0 : mu;
            sh.inv = raw ? 1.0 : var <= 1e-24 * (mm > 1.0 ? mm : 1.0) ? 0.0 : 1.0 / sqrt(var);
        }
    }
    group_bar(bar, kFxThreads);
    const double mu = sh.mu, inv = sh.inv;
    for (int j = t; j < m; j += kFxThreads) cd[j] = df_from(((double)xw[j] - mu) * inv);
    group_bar(bar, kFxThreads);
}

}  // namespace dtws
