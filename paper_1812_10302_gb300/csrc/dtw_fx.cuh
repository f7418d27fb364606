// dtw_fx.cuh -- the extended-precision banded DTW of one window as fast as one
// CTA can walk it: 64-bit fixed-point path sums, costs formed by other warps.
#pragma once

#include "dtw_band.cuh"

namespace dtws {

// One window's re-score is pure latency: 2m - 1 dependent anti-diagonals.  In
// double-float (dtw_diag_df) a step costs ~41 instructions per cell, most of
// them the cell's cost, and one warp issued them all: 262 cycles per step at
// r = 51.  Three things split the work.
//   * Producer warps form the costs (q_hat_i - c_j)^2 of the coming
//     anti-diagonals in double-float, as before, turn each into a 64-bit
//     integer and leave it in a shared-memory ring; consumer warps walk: per
//     cell two integer minima and one addition (10 instructions), per step one
//     neighbour exchange by shuffle.  The two halves meet at a named barrier
//     every chunk of anti-diagonals.
//   * Integer sums do not depend on their order, so the matrix is walked from
//     both ends at once, by the two CTAs of a cluster (the second one on the
//     reversed sequences), and the best path is the best way of joining the
//     two middle anti-diagonals: half the steps, the same result to the bit.
//   * Bands past one warp's cells (four a lane: r > 126) take W consumer warps
//     whose cells overlap by one lane on each side.  In kFxUnit = 8 steps an
//     error at a warp's edge travels four cells, one lane; then the overlap is
//     taken anew from the neighbours (one exchange per chunk).
//   * With six such warps and more the producers beside them take more issue
//     slots than the walk: a second CTA per direction forms most of the costs
//     and writes them into the walking CTA's ring (distributed shared memory).
//     m = 1024, r = 921, whole call: 302 us, 428 with two CTAs to a cluster; at
//     W = 2 to 4 the cluster's barrier per chunk costs more than that (m = 2048,
//     r = 200 403 us, 305 without).
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
// Measured, dtws_dtw_at_f64 of one window, whole call: 76 us at m = 512,
// r = 51 (105 us walked from one end, 164 us in double-float), 132 us at
// m = 1024, r = 102 (210, 412), 170 us at r = 200 (311, 513); bound by the
// consumers' ALU issue (25 cycles per cell of a lane) past two cells per lane,
// and on several warps by the producers' beside it.
constexpr int kFxUnit = 8, kFxRMax = 1023;
// a saturated cost; the value saturated sums are set back to every kFxUnit
// steps (kFxInf + kFxUnit * kFxCost < 2^64, so no sum wraps in between)
constexpr unsigned long long kFxCost = 1ull << 60, kFxInf = 1ull << 61, kFxRedo = 1ull << 51;

// A walk's shape: K cells per lane, W consumer warps.
template <int K_, int W_>
struct Fx {
    static constexpr int K = K_, W = W_;
    static constexpr int kThreads = W == 1 ? 384 : 768, kWarps = kThreads / 32;
    static constexpr int kCtas = W < 6 ? 2 : 4;  // of a cluster: two that walk, past W = 4 two that only form costs
    static constexpr int kSteps = W == 1 ? 16 : kFxUnit;   // anti-diagonals of a chunk
    static constexpr int kLanes = W == 1 ? 32 : 30 * W + 2;  // lanes without the overlaps
    static constexpr int kCells = K * kLanes;
    static constexpr int kStep = ((K + 1) / 2) * kLanes * 2;  // words of a step in the ring
    static constexpr size_t kRing = (size_t)2 * kSteps * kStep * 8;
    static_assert(W == 1 || K == 4, "an overlap is one lane and lasts kFxUnit steps");
};

// kCells >= r + 2, so the last cell of every anti-diagonal lies past the band
// and is always saturated: the neighbour exchange may then wrap around the
// warp without a special case at the upper end.
#define DTWS_FX_SHAPES(X) X(1, 1) X(2, 1) X(3, 1) X(4, 1) X(4, 2) X(4, 3) X(4, 4) X(4, 6) X(4, 9)
struct FxPlan {
    int K, W, threads;
    size_t ring;
};
__host__ __device__ inline FxPlan fx_plan(int r) {
#define DTWS_FX_TRY(KK, WW) \
    if (Fx<KK, WW>::kCells >= r + 2) return FxPlan{KK, WW, Fx<KK, WW>::kThreads, Fx<KK, WW>::kRing};
    DTWS_FX_SHAPES(DTWS_FX_TRY)
#undef DTWS_FX_TRY
    return FxPlan{0, 0, 0, 0};
}
// Padding on each side of the query's and the window's double-floats: a
// producer's positions run to r/2 + 1 before either start and, on the last
// chunk's steps past the middle, at most 12 past either end.
__host__ __device__ inline int fx_pad(int r) { return ((r >> 1) + 20) & ~1; }
__host__ __device__ inline size_t fx_span(int m, int r) { return (size_t)((m + 2 * fx_pad(r) + 1) & ~1); }
// shared memory of one window: the ring, the query's and the window's padded double-floats
__host__ __device__ inline size_t fx_bytes(int m, int r) { return fx_plan(r).ring + fx_span(m, r) * 16; }
// whether a search re-scores with this walk: one rule for the pre-score and
// the final stage, so that equal windows are compared on equal terms
__host__ __device__ inline bool fx_used(int m, int r) {
    return r <= kFxRMax && fx_bytes(m, r) <= (size_t)216 * 1024;
}

struct FxShared {
    float red[24];
    unsigned long long res;
    ulonglong2 edge[2][9][2][4];  // [chunk parity][warp][lower, upper edge][p1's two pairs, p2's two pairs]
    double mu, inv;
};

// The cluster's barrier and its peer's shared memory.
__device__ __forceinline__ int cluster_rank() {
    int v;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
    return v;
}
__device__ __forceinline__ void cluster_bar() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned peer_addr(const void *p, int rank) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), v;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(v) : "r"(a), "r"(rank));
    return v;
}
__device__ __forceinline__ unsigned long long peer_load(unsigned a) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void peer_store(unsigned a, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

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
// far: the ring of the cluster's CTA `rank` instead of this one's (dst: this
// one's address of the slots).
template <typename S>
__device__ __forceinline__ void fx_produce(const dfloat *qd, const dfloat *cd, int r, float f, int v0, int blk,
                                           unsigned long long *dst, int lane, bool far, int rank) {
    const int p = blk * 32 + lane, a = v0 - (r & 1);
    if (S::kCells % 32 && p >= S::kCells) return;
    const int pc = p < r ? p : r;  // (past the band no cost counts, and no address either)
    const dfloat *qp = qd + (((a + r) >> 1) - pc), *cp = cd + (((a - r) >> 1) + pc);
    const int pl = p / S::K, pt = p - pl * S::K;
    unsigned long long *o = dst + ((pt >> 1) * S::kLanes + pl) * 2 + (pt & 1);
    const unsigned oa = far ? peer_addr(o, rank) : 0u;
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
            const unsigned long long w = fx_round(sq, er), v = fine ? w : kFxCost;
            if (S::kCtas > 2 && far) peer_store(oa + (s + e) * S::kStep * 8, v);
            else o[(s + e) * S::kStep] = v;
        }
    }
}

// One anti-diagonal of the walk: cell t of the lane (as diag_step).  vl: the
// lane's place on the anti-diagonal.
template <typename S, int ODD>
__device__ __forceinline__ void fx_step(const unsigned long long *buf, unsigned long long (&p1)[S::K],
                                        unsigned long long (&p2)[S::K], int lane, int vl) {
    constexpr int K = S::K;
    unsigned long long cost[((K + 1) / 2) * 2];
#pragma unroll
    for (int t = 0; t < (K + 1) / 2; ++t) {
        const ulonglong2 c = reinterpret_cast<const ulonglong2 *>(buf)[t * S::kLanes + vl];
        cost[2 * t] = c.x;
        cost[2 * t + 1] = c.y;
    }
    unsigned long long nb =
        __shfl_sync(0xffffffffu, ODD ? p1[0] : p1[K - 1], ODD ? ((lane + 1) & 31) : ((lane - 1) & 31));
    if (S::W > 1 && !ODD) nb = vl == 0 ? kFxInf : nb;  // (the first warp's last lane is not the band's end)
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

// The walk by the S::kThreads threads of each of a cluster's CTAs (all of
// them).  rank: the CTA's; its lowest bit is the direction, 1 for the reversed
// sequences; ranks 2 and 3 only form costs.  qd, cd:
// element 0 of q_hat and of the normalised window as double-floats (reversed
// in direction 1), padded by fx_pad(r) elements of +1e15 and -1e15 on both
// sides; bound: an upper bound of the DTW, 0 for the diagonal path's cost;
// ring: S::kRing bytes, 16-byte aligned.  Every thread of all CTAs returns
// the distance.
template <typename S>
__device__ double dtw_fx(const dfloat *__restrict__ qd, const dfloat *__restrict__ cd, int m, int r, float bound,
                         int rank, FxShared &sh, unsigned long long *ring) {
    constexpr int K = S::K, W = S::W;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, dir = rank & 1;
    const bool helper = rank >= 2;  // (forms costs for the ring of rank - 2)
    // A helper's first act is a store into its walker's shared memory, which
    // may only be touched once every CTA of the cluster is known to have
    // started.  (With two CTAs the first access comes after a chunk's meeting
    // and the join's barrier.)
    if constexpr (S::kCtas > 2) cluster_bar();
    // the diagonal path's cost, an upper bound of the DTW (the same sum, in
    // the same order, in every thread of all CTAs)
    auto euclid = [&]() {
        float ed = 0.0f;
        for (int j = t; j < m; j += S::kThreads) {
            const int i = dir ? m - 1 - j : j;
            const float d = df_sub(qd[i], cd[i]).hi;
            ed = fmaf(d, d, ed);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ed += __shfl_xor_sync(0xffffffffu, ed, o);
        if (lane == 0) sh.red[warp] = ed;
        __syncthreads();
        ed = 0.0f;
#pragma unroll
        for (int w = 0; w < S::kWarps; ++w) ed += sh.red[w];
        __syncthreads();  // (sh.red is read before it is written again)
        return ed;
    };
    auto scale_of = [](float bound) { return (58 - (ilogbf(bound * 1.001f) + 1)) >> 1; };
    if (!(bound > 0.0f && bound < 1e30f)) bound = euclid();
    if (!(bound > 0.0f)) return 0.0;  // (the Euclidean distance is 0)
    int h = scale_of(bound);          // the scale is 2^(2h)
    // the forward walk ends on anti-diagonal m - 1, the reversed one on the
    // next (its own m - 2)
    const int V = m - dir + (r & 1);
    // (the directions meet at every chunk where the cluster's barrier ends it:
    // as many for both then)
    const int chunks = ((S::kCtas > 2 ? m + (r & 1) : V) + S::kSteps - 1) / S::kSteps;
    const bool walks = warp < W && !helper;
    // a chunk ends where its walkers and producers meet
    auto meet = []() {
        if constexpr (S::kCtas > 2) cluster_bar();
        else __syncthreads();
    };
    const int p0 = (r - (r & 1)) >> 1;
    const int vl = W == 1 ? lane : warp * 30 + lane;
    // the lanes whose cells are this warp's own
    const bool own = walks && (warp == 0 || lane > 0) && (warp == W - 1 || lane < 31);
    for (int pass = 0;; ++pass) {
        const float f = ldexpf(1.0f, h);
        // a chunk's units: kFxUnit steps of one block of 32 cells each, of the
        // blocks that hold cells of the band; the others' costs never change
        constexpr int kBlks = (S::kCells + 31) / 32;
        const int blks = S::kCtas == 2 ? kBlks : r / 32 + 1;  // (two CTAs: no division by a variable)
        auto produce = [&](int c, int w, int nw) {
            unsigned long long *buf = ring + (size_t)(c & 1) * S::kSteps * S::kStep;
            for (int u = w; u < blks * (S::kSteps / kFxUnit); u += nw) {
                const int blk = u % blks, s0 = u / blks * kFxUnit;
                fx_produce<S>(qd, cd, r, f, c * S::kSteps + s0, blk, buf + s0 * S::kStep, lane, helper, dir);
            }
        };
        if constexpr (S::kCtas > 2) {
            for (int p = blks * 32 + t; p < S::kCells && !helper; p += S::kThreads) {
                const int pl = p / K, pt = p - pl * K;
                for (int s = 0; s < 2 * S::kSteps; ++s)
                    ring[(size_t)s * S::kStep + ((pt >> 1) * S::kLanes + pl) * 2 + (pt & 1)] = kFxCost;
            }
        }
        // the helper's warps first, then the ones that don't walk
        const int pw = S::kCtas == 2 ? warp - W : helper ? warp : S::kWarps + warp - W;
        constexpr int kPw = S::kCtas == 2 ? S::kWarps - W : 2 * S::kWarps - W;
        if constexpr (S::kCtas == 2) produce(0, warp, S::kWarps);
        else if (!walks) produce(0, pw, kPw);
        meet();
        unsigned long long p1[K], p2[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
            // the base cell lies on anti-diagonal -2: two steps before v = 0
            // when r is even, one before when r is odd
            const unsigned long long base = vl * K + u == p0 ? 0ull : kFxInf;
            p1[u] = (r & 1) ? base : kFxInf;
            p2[u] = (r & 1) ? kFxInf : base;
        }
        for (int c = 0; c < chunks; ++c) {
            const unsigned long long *buf = ring + (size_t)(c & 1) * S::kSteps * S::kStep;
            if (walks) {
                const int steps = V - c * S::kSteps < S::kSteps ? V - c * S::kSteps : S::kSteps;  // (0: none left)
                if (steps == S::kSteps) {
#pragma unroll 1
                    for (int s0 = 0; s0 < S::kSteps; s0 += kFxUnit) {
#pragma unroll
                        for (int s = s0; s < s0 + kFxUnit; s += 2) {
                            fx_step<S, 0>(buf + s * S::kStep, p1, p2, lane, vl);
                            fx_step<S, 1>(buf + (s + 1) * S::kStep, p1, p2, lane, vl);
                        }
                        fx_clamp<K>(p1);
                        fx_clamp<K>(p2);
                    }
                } else {
                    for (int s = 0; s < steps; s += 2) {
                        fx_step<S, 0>(buf + s * S::kStep, p1, p2, lane, vl);
                        if (s + 1 < steps) fx_step<S, 1>(buf + (s + 1) * S::kStep, p1, p2, lane, vl);
                        if ((s + 2) % kFxUnit == 0) {
                            fx_clamp<K>(p1);
                            fx_clamp<K>(p2);
                        }
                    }
                }
                if constexpr (W > 1) {  // the own cells beside each overlap
                    if (lane == 1 || lane == 30) {
                        ulonglong2 *e = sh.edge[c & 1][warp][lane == 30];
                        e[0] = make_ulonglong2(p1[0], p1[1]);
                        e[1] = make_ulonglong2(p1[2], p1[3]);
                        e[2] = make_ulonglong2(p2[0], p2[1]);
                        e[3] = make_ulonglong2(p2[2], p2[3]);
                    }
                }
            } else if (c + 1 < chunks) {
                produce(c + 1, pw, kPw);
            }
            meet();
            if constexpr (W > 1) {
                if (walks && ((lane == 0 && warp > 0) || (lane == 31 && warp < W - 1))) {
                    const ulonglong2 *e = lane == 0 ? sh.edge[c & 1][warp - 1][1] : sh.edge[c & 1][warp + 1][0];
                    const ulonglong2 a0 = e[0], a1 = e[1], b0 = e[2], b1 = e[3];
                    p1[0] = a0.x;
                    p1[1] = a0.y;
                    p1[2] = a1.x;
                    p1[3] = a1.y;
                    p2[0] = b0.x;
                    p2[1] = b0.y;
                    p2[2] = b1.x;
                    p2[3] = b1.y;
                }
                __syncwarp();
            }
        }
        // The join.  The reversed walk's cell p' of an even (odd) step is the
        // forward one's r - p' (r - 1 - p').  A path goes through
        // anti-diagonal m - 1 (p1) and then m or, diagonally, m + 1, or from
        // m - 2 (p2) diagonally to m.
        fx_clamp<K>(p1);
        fx_clamp<K>(p2);
        unsigned long long *last1 = ring, *last2 = ring + S::kCells;
        if (t == 0) sh.res = ~0ull;
        if (dir && own) {
#pragma unroll
            for (int u = 0; u < K; ++u) {
                last1[vl * K + u] = p1[u];
                last2[vl * K + u] = p2[u];
            }
        }
        cluster_bar();
        if (!dir && walks) {
            const bool even = ((m - 1 + r) & 1) == 0;  // anti-diagonal m - 1 is an even step
            const unsigned a1 = peer_addr(last1, 1), a2 = peer_addr(last2, 1);
            auto at = [](unsigned a, int j) { return j >= 0 ? peer_load(a + (unsigned)j * 8) : kFxInf; };
            const int j1 = (even ? r - 1 : r) - vl * K, j2 = (even ? r : r - 1) - vl * K;
            unsigned long long best = ~0ull;
            if (own) {
                // anti-diagonal m: the cells beside cell u are u - 1 and u
                // when m - 1 is an even step, u and u + 1 when it is odd
                unsigned long long n[K + 1];
#pragma unroll
                for (int u = 0; u <= K; ++u) {
                    const int p = vl * K + u - (even ? 1 : 0);
                    n[u] = p >= 0 ? at(a1, j1 - (p - vl * K)) : kFxInf;
                }
#pragma unroll
                for (int u = 0; u < K; ++u) {
                    const unsigned long long d = even ? n[u + 1] : n[u];
                    best = fx_min(best, p1[u] + fx_min(fx_min(n[u], n[u + 1]), at(a2, j2 - u)));
                    best = fx_min(best, p2[u] + d);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = fx_min(best, __shfl_xor_sync(0xffffffffu, best, o));
            if (lane == 0) atomicMin(&sh.res, best);
        }
        __syncthreads();
        if (rank == 0 && t > 0 && t < S::kCtas) peer_store(peer_addr(&sh.res, t), sh.res);
        cluster_bar();
        const unsigned long long res = sh.res;
        __syncthreads();  // (sh.res is read before it is written again)
        if (res > (1ull << 59) && pass < 3) {  // `bound` did not hold: the Euclidean distance does
            bound = euclid();
            h = scale_of(bound);
            continue;
        }
        if (res >= kFxRedo || pass >= 3) return ldexp((double)res, -2 * h);
        // a DTW far below the bound: again on its own scale (its 2 m - 1
        // roundings allowed for), which puts it below 2^57; never past what
        // FP32 scales by (2^(2 * 120))
        const int up = (56 - (63 - __clzll((long long)(res + 2 * m)))) >> 1;
        if (h + up > 120) return ldexp((double)res, -2 * h);
        h += up;
    }
}

template <typename S>
__device__ __forceinline__ void fill_pads_fx(dfloat *base, int m, int pad, dfloat v) {
    for (int u = threadIdx.x; u < 2 * pad; u += S::kThreads) base[u < pad ? u : m + u] = v;
}

// The padded query and window copies behind the ring, their pads poisoned and
// the query filled (reversed when dir is 1), by the CTA's threads (the next
// barrier, in fx_window, makes them visible).
template <typename S>
__device__ __forceinline__ void fx_setup(unsigned char *sm, const double *__restrict__ qh64, int m, int r, int dir,
                                         dfloat **qd, dfloat **cd) {
    const int pad = fx_pad(r);
    dfloat *q = (dfloat *)(sm + S::kRing), *c = q + fx_span(m, r);
    fill_pads_fx<S>(q, m, pad, dfloat{1e15f, 0.0f});
    fill_pads_fx<S>(c, m, pad, dfloat{-1e15f, 0.0f});
    for (int j = threadIdx.x; j < m; j += S::kThreads) q[pad + (dir ? m - 1 - j : j)] = df_from(qh64[j]);
    *qd = q + pad;
    *cd = c + pad;
}

// Two-pass FP64 statistics (Eq. 5) of the window xw by the CTA's first warp
// into sh.mu, sh.inv (0 under the zero-variance rule; 0 and 1 for raw
// values), then its normalised values as double-floats (reversed when dir is
// 1).  All threads of the CTA call it; they have met at the barrier on return.
template <typename S>
__device__ __forceinline__ void fx_window(const float *__restrict__ xw, int m, bool raw, int dir, dfloat *cd,
                                          FxShared &sh) {
    const int t = threadIdx.x, lane = t & 31;
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
    __syncthreads();
    const double mu = sh.mu, inv = sh.inv;
    for (int j = t; j < m; j += S::kThreads) cd[dir ? m - 1 - j : j] = df_from(((double)xw[j] - mu) * inv);
    __syncthreads();
}

}  // namespace dtws
