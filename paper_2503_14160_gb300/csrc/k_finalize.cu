// The last part of Algorithm 1 step (2): per candidate, the FP64 sums of its work items
// (J_p, the penetration sum, J_l, the path length, and the count of checkpoints in
// collision) added in item order into J = J_p + w_c lambda_c sum_k pen_k + w_l J_l
// (Eq. path opt; arXiv 2503.14160, Sec. 4.1). The order of the additions is fixed, so results
// are deterministic.
//
// Four lanes per candidate, one per sum, so that a candidate's loads are whole 32-byte sectors
// and eight items' loads are in flight before the dependent FP64 additions (each holds a
// scheduler's FP64 unit for some 70 cycles whatever its lanes do) take them in item order. The
// kernel is bound by the latency of one such chain (256 candidates of 32 checkpoints per span: 7.8 us
// with one thread per candidate, 4.4 with four).
#include "chain_launch.cuh"
#include "cp_internal.cuh"

namespace cp {
namespace {

constexpr int kFinalLanes = 4;    // lanes per candidate
constexpr int kFinalAhead = 8;    // items loaded ahead

// Candidate i on the kFinalLanes aligned lanes that share it (sub = lane within the group).
// Called by whole warps.
__device__ __forceinline__ void finalize_body(const double *item_sum,
                                              const uint32_t *item_count, int n, int P, double w_c,
                                              double w_l, double lambda_c, double *J, uint8_t *flag, double *terms,
                                              const uint32_t *status, int i, int sub)
{
    double acc = 0.0;
    uint32_t n_flagged = 0;
    if (i < n) {
        const double *row = item_sum + (size_t)i * P * 4 + sub;
        const uint32_t *crow = item_count + (size_t)i * P;
        for (int p0 = 0; p0 < P; p0 += kFinalAhead) {
            double v[kFinalAhead];
#pragma unroll
            for (int q = 0; q < kFinalAhead; ++q) v[q] = p0 + q < P ? row[4 * (p0 + q)] : 0.0;
#pragma unroll
            for (int q = 0; q < kFinalAhead; q += kFinalLanes)
                if (p0 + q + sub < P) n_flagged += crow[p0 + q + sub];
#pragma unroll
            for (int q = 0; q < kFinalAhead; ++q)
                if (p0 + q < P) acc += v[q];
        }
    }
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int off = 1; off < kFinalLanes; off <<= 1) n_flagged += __shfl_xor_sync(full, n_flagged, off);
    const int lead = (int)(threadIdx.x & 31) & ~(kFinalLanes - 1);
    double jp = __shfl_sync(full, acc, lead), jc = __shfl_sync(full, acc, lead + 1);
    double jl = __shfl_sync(full, acc, lead + 2), len = __shfl_sync(full, acc, lead + 3);
    if (i >= n || sub != 0) return;
    jc *= lambda_c;
    double Ji = jp + w_c * jc + w_l * jl;
    uint8_t fl = n_flagged > 0 ? 1 : 0;
    if (status != nullptr && *status != 0u) {
        // the evaluation gave up on a bounded wait: some item sums are stale, so no result
        // of this call is valid (NaN cost, flagged)
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        jp = jc = jl = len = Ji = nan;
        fl = 1;
    }
    J[i] = Ji;
    if (flag != nullptr) flag[i] = fl;
    if (terms != nullptr) {
        double *tm = terms + (size_t)i * 5;
        tm[0] = jp;
        tm[1] = jc;
        tm[2] = jl;
        tm[3] = len;
        tm[4] = (double)n_flagged;
    }
}

__global__ void __launch_bounds__(256)
k_eval_finalize(const double *item_sum, const uint32_t *item_count, int n, int P,
                double w_c, double w_l, double lambda_c, double *J, uint8_t *flag, double *terms,
                const uint32_t *status, int *queue)
{
    after_previous();
    if (queue != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *queue = 0;
    const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    finalize_body(item_sum, item_count, n, P, w_c, w_l, lambda_c, J, flag, terms, status, t / kFinalLanes,
                  t % kFinalLanes);
}

// Every query's costs in one launch: block b of query q takes its candidates 256 b .. with
// 1024 threads; the mean form takes the single mean candidate of query blockIdx.x (with the
// terms) on one warp.
__global__ void __launch_bounds__(256 * kFinalLanes)
k_batch_finalize(const BatchQueryDev *__restrict__ qd, const int2 *__restrict__ tab, const BatchEvalDev *ev)
{
    if (tab != nullptr) {
        const int2 e = tab[blockIdx.x];
        const BatchQueryDev &q = qd[e.x];
        finalize_body(q.item_sum, q.item_count, q.N, q.P, q.w_c, q.w_l, q.lambda_c, q.J, q.flag, nullptr, nullptr,
                      e.y * 256 + (int)threadIdx.x / kFinalLanes, (int)threadIdx.x % kFinalLanes);
    } else {
        const BatchQueryDev &q = qd[blockIdx.x];
        const EvalArgs &a = ev[blockIdx.x].a;
        finalize_body(a.item_sum, a.item_count, 1, a.P, q.w_c, q.w_l, q.lambda_c, q.mean_J, q.mean_flag,
                      q.mean_terms, nullptr, (int)threadIdx.x / kFinalLanes, (int)threadIdx.x % kFinalLanes);
    }
}

}  // namespace

int launch_eval_finalize(const double *item_sum, const uint32_t *item_count, int n, int P,
                         double w_c, double w_l, double lambda_c, double *J, uint8_t *flag,
                         double *terms, cudaStream_t st, const uint32_t *status, int *queue)
{
    if (n == 0) return CP_OK;
    const int threads = 256, per = threads / kFinalLanes;
    launch_chained(k_eval_finalize, (unsigned)((n + per - 1) / per), threads, 0, st, item_sum, item_count, n, P, w_c,
                   w_l, lambda_c, J, flag, terms, status, queue);
    CP_LAUNCHED("k_eval_finalize");
    return CP_OK;
}

int launch_batch_finalize(const BatchQueryDev *qd, const int2 *tab, int blocks, const BatchEvalDev *mean_ev,
                          cudaStream_t st)
{
    if (blocks == 0) return CP_OK;
    k_batch_finalize<<<blocks, tab != nullptr ? 256 * kFinalLanes : 32, 0, st>>>(qd, tab, mean_ev);
    CP_LAUNCHED("k_batch_finalize");
    return CP_OK;
}

}  // namespace cp
