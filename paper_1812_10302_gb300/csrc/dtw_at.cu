// dtw_at.cu -- FP32 banded DTW at given offsets of a handle's series
// (dtw_at.cuh).
#include "dtw_at.cuh"

namespace dtws {

namespace {

template <int L, int K>
__global__ void __launch_bounds__(kAtThreads, at_min_blocks(K))
k_dtw_at(QueryBufs b, QueryArgs a, const int64_t *__restrict__ offsets, int64_t count, float *__restrict__ out) {
    if (!b.st->valid) return;
    at_body<L, K>(b.qh32, b.x, a.N, a.m, a.r, offsets, count, out,
                  [&](int64_t o, int, unsigned, float &mh, float &is, float &ls) {
                      mh = b.mu_hi[o];
                      is = b.inv_sigma[o];
                      ls = b.mu_lo[o] * is;
                  });
}

template <int L, int K>
cudaError_t at_launch(const QueryBufs &b, const QueryArgs &a, const int64_t *offsets, int64_t count, float *out,
                      const AtPlan &p, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_dtw_at<L, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e != cudaSuccess) return e;
    k_dtw_at<L, K><<<at_grid(p, count, b.num_sms), p.warps * 32, p.smem, s>>>(b, a, offsets, count, out);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dtw_at_many(const QueryBufs &b, const QueryArgs &a, const int64_t *offsets, int64_t count, float *out,
                               cudaStream_t s) {
    AtPlan p;
    if (!at_plan(a.m, a.r, &p)) return cudaErrorNotSupported;
#define DTWS_CASE(LL, KK) \
    if (p.L == LL && p.K == KK) return at_launch<LL, KK>(b, a, offsets, count, out, p, s);
    DTWS_AT_SHAPES(DTWS_CASE)
#undef DTWS_CASE
    return cudaErrorInvalidValue;
}

}  // namespace dtws
