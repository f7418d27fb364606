// dtw_at.cuh -- FP32 banded DTW at given offsets: the walk of dtw_band.cuh
// arranged for the grid's rate (every walk runs to its end, so one walk's
// latency does not count).
#pragma once

#include "dtw_band.cuh"
#include "dtws_internal.h"

namespace dtws {

// dtw_diag is bound by instruction issue: per cell a subtraction, a
// multiply-add, a three-input minimum and half a band mask, per anti-diagonal
// and lane ~6 for the neighbour exchange and the register windows.  Per pair of
// anti-diagonals and lane 7 K + 12 instructions, so a window costs
// L (7 K + 12) per pair on L lanes of K cells (6 fewer with an odd K, whose lanes
// load their own register windows, and a spare cell): few lanes with many cells, and
// as few cells past the band as the shapes allow.  At r = 51 (52 cells) eight
// lanes of seven cells cost 440 where 16 x 4 cost 640.  Measured (1e5 windows,
// m = 512, r = 51; 25,000, m = 1024, r = 102; 3e5, m = 128, r = 12): 0.86, 0.89
// and 0.21 ms, against 1.04, 1.07 and 0.42 on (16, 4), (32, 4) and (8, 2).
// (Two windows per lane in packed FP32 pairs, 9 K + 17 instructions for both,
// were no faster: the packed operations stall the dispatch, 55 % issue, and
// two windows per group halve the warps that fit.)
// Shapes: X(L, K): those that at_plan takes for some length up to 8192 and
// some band (never 8 or 16 lanes of 6 cells: it was tried for all of them).
#define DTWS_AT_SHAPES(X)                                                                                 \
    X(2, 4) X(2, 5) X(2, 7) X(4, 3) X(4, 4) X(4, 5) X(4, 6) X(4, 7) X(4, 8) X(8, 3) X(8, 4) X(8, 5) X(8, 7) \
    X(8, 8) X(16, 3) X(16, 4) X(16, 5) X(16, 7) X(16, 8) X(32, 3) X(32, 4) X(32, 5) X(32, 6) X(32, 7) X(32, 8)
constexpr int kAtThreads = 256;
constexpr size_t kAtSmemMax = (size_t)224 * 1024;  // of an SM, and of a CTA at most
// resident CTAs the register bound is set for
__host__ __device__ constexpr int at_min_blocks(int K) { return K <= 3 ? 4 : 3; }

// (congruent to L modulo the 32 banks: with an odd K the lanes of all the
// groups of a warp then load from different banks)
__host__ __device__ inline size_t at_span(int m, int r, int L, int K) {
    return (size_t)((m + 2 * diag_pad(r, L, K) + 31 - L) / 32 * 32 + L);
}
struct AtPlan {
    int L, K, warps, per_sm;
    size_t smem;
};
// The shape for (m, r): the least cost * (w + 5) / w among the shapes with
// L K >= r + 2, w the warps their window copies leave on an SM: few warps hide
// less of a step's latency (a band far narrower than the query stages many
// long windows per warp).  The 5 fits a sweep of every shape at 14 sizes, m =
// 128..8192, r = 12..250: e.g. (before the odd shapes' own loads) m = 512,
// r = 51 0.92 ms for (8, 7) on 18 warps and 1.07 for (16, 4) on 32; m = 1024, r = 20 0.65 ms for (8, 3) on 12 warps,
// 0.72 for (4, 6) on 6 and 1.17 for (16, 3) on 20; more than eight cells per
// lane never won.  False: bands of fewer than 5 or more than 256 cells (the
// walks of k_dtw), or copies that do not fit.
inline bool at_plan(int m, int r, AtPlan *best) {
    const int need = r + 1;
    if (need < 5 || need > 256) return false;
    bool found = false;
    double best_score = 0.0;
#define DTWS_AT_TRY(LL, KK)                                                                            \
    if (LL * KK > need) {                                                                             \
        const size_t span = at_span(m, r, LL, KK) * 4, per = (size_t)(32 / LL) * span;                 \
        const int blocks = at_min_blocks(KK);                                                          \
        int warps = kAtThreads / 32;                                                                   \
        while (warps > 1 && span + (size_t)warps * per > kAtSmemMax / blocks) --warps;                 \
        const size_t total = span + (size_t)warps * per;                                               \
        int on_sm = (int)(kAtSmemMax / total); /* (0: no warp's copies fit) */                         \
        if (on_sm > blocks) on_sm = blocks;                                                            \
        const int w = on_sm * warps;                                                                   \
        const double score = w > 0 ? LL * (7 * KK + ((KK & 1) ? 6 : 10)) * (w + 5.0) / w : 0.0;                         \
        if (w > 0 && (!found || score < best_score)) {                                                 \
            found = true;                                                                              \
            best_score = score;                                                                        \
            *best = AtPlan{LL, KK, warps, on_sm, total};                                               \
        }                                                                                              \
    }
    DTWS_AT_SHAPES(DTWS_AT_TRY)
#undef DTWS_AT_TRY
    return found;
}

// A kernel's body: the window at offsets[c] by group c, c + groups, ...  (every
// walk costs the same: nothing to balance).  stats(o, lane, gmask, mh, is, ls):
// the window's normalisation, by the group's lanes, the same in each.
// Offsets outside [0, N) give NaN.
template <int L, int K, typename Stats>
__device__ __forceinline__ void at_body(const float *__restrict__ qh, const float *__restrict__ x, int64_t N, int m,
                                        int r, const int64_t *__restrict__ offsets, int64_t count,
                                        float *__restrict__ out, Stats &&stats) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const float INF = __int_as_float(0x7f800000);
    const int pad = diag_pad(r, L, K);
    float *qs = (float *)smraw + pad;
    for (int t = threadIdx.x; t < m; t += blockDim.x) qs[t] = qh[t];
    for (int t = threadIdx.x; t < 2 * pad; t += blockDim.x) qs[t < pad ? t - pad : m + t - pad] = INF;
    const int ln = lane_id(), g = ln / L, lane = ln % L;
    const int gid = (int)(threadIdx.x >> 5) * (32 / L) + g;
    const unsigned gmask = (L == 32) ? 0xffffffffu : (((1u << L) - 1u) << (g * L));
    float *cs = (float *)smraw + (size_t)(1 + gid) * at_span(m, r, L, K) + pad;
    for (int t = lane; t < 2 * pad; t += L) cs[t < pad ? t - pad : m + t - pad] = -INF;
    __syncthreads();
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x / L);
    for (int64_t c = (int64_t)blockIdx.x * (blockDim.x / L) + gid; c < count; c += groups) {
        const int64_t o = offsets[c];
        if (o < 0 || o >= N) {
            if (lane == 0) out[c] = __int_as_float(0x7fc00000);
            continue;
        }
        float mh, is, ls;
        stats(o, lane, gmask, mh, is, ls);
        const float *xw = x + o;
        __syncwarp(gmask);  // (the previous walk's reads come before these writes)
        for (int j = lane; j < m; j += L) cs[j] = fmaf(xw[j] - mh, is, -ls);
        __syncwarp(gmask);
        int cells = 0;
        const float d = dtw_diag<float, L, K, false, true>(qs, cs, nullptr, 0.0f, m, r, INF, gmask, lane, cells);
        if (lane == 0) out[c] = d;
    }
}

// Grid of a launch of `count` windows.
inline unsigned at_grid(const AtPlan &p, int64_t count, int num_sms) {
    const int per_cta = p.warps * (32 / p.L);
    const int64_t want = (count + per_cta - 1) / per_cta, cap = (int64_t)num_sms * p.per_sm;
    return (unsigned)(want < cap ? want : cap);
}

}  // namespace dtws
