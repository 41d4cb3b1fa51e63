// The Cholesky factor of the sampling distribution, L L^T = sigma^2 C in FP64 (Algorithm 1 step
// (1); arXiv 2503.14160, Sec. 4.1), D = 4K <= 128, as a dataflow over a thread-block cluster.
//
// What bounds it. An FP64 warp instruction holds its scheduler's FP64 unit for 64 cycles, and a
// dependent one waits as long, so one SM needs 350k cycles for the D^3 / 6 FMAs of D = 128, and
// a column's chain (t = a d, the next pivot, its reciprocal) about 550 cycles on any number of
// SMs. One CTA that took the columns in turn with two block barriers each needed 1400-1900
// cycles per column (ncu: 24 us at D = 32, 56 at 64, 198 at 128).
//
// The form is the right-looking L D L^T one: column k takes t_i = a_ik / a_kk for the rows below
// the pivot and a_ij -= t_i a_jk, so every entry receives its updates in ascending k, one FMA
// each: the split below does not change a bit. CTA b of the cluster owns rows 16 b .. 16 b + 15
// and keeps them in shared memory (a warp instruction holds 16 rows x 2 neighbouring columns, the
// column pairs dealt to the warps; in registers the pairs that are finished cost their FP64
// instruction all the same, as the compiler makes the choice by selects). Row i needs column k of
// rows j <= i only, so data flows one way, from a CTA to the later ones: before step k a CTA sends
// its 16 entries of column k, and the owner of pivot k also sends 1 / a_kk and a_kk, by st.async into the receivers' shared memory, which
// completes on the receivers' mbarrier of column k. Within its own 16 columns a CTA has the
// pivots to itself: warp 0 works one column ahead on the reciprocal, on the scheduler that has
// one worker warp instead of two, while the workers apply the current column; one block barrier
// per column. Each wait for another CTA has a limit and ends in DEV_ERR_TIMEOUT.
//
// Measured (factor and the two small copies of cp_set_distribution): 31.6 -> 24.8 us at D = 32,
// 62.9 -> 41.4 at 64, 116.9 -> 62.9 at 96, 201.4 -> 87.9 at 128. An own column takes 870 cycles:
// the pivot's chain of 550, the shared-memory round trips and the block barrier; the last CTA's early
// columns, with up to 64 pairs, 1300 on average.
#include <atomic>

#include <cooperative_groups.h>

#include "chain_launch.cuh"
#include "cp_internal.cuh"
#include "fp64_chain.cuh"
#include "tcgen05.cuh"

namespace cp {
namespace {

constexpr int kRows = 16;                               // rows per CTA
constexpr int kFactorThreads = 256;
constexpr int kWarps = kFactorThreads / 32;             // all work on the earlier CTAs' columns;
constexpr int kWorkers = kWarps - 1;                    // on the own ones warp 0 takes the pivots
constexpr int kMaxFactorD = 4 * CP_MAX_WAYPOINTS;
constexpr int kMaxCtas = kMaxFactorD / kRows;           // 8: a portable cluster
constexpr long long kFactorWaitCycles = 2000000000ll;   // about one second

__device__ __forceinline__ uint32_t remote_addr(const void *p, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(tc::smem_addr(p)), "r"(rank));
    return r;
}

__device__ __forceinline__ void send_double(const double *dst, uint64_t *bar, int rank, double v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
                 :: "r"(remote_addr(dst, rank)), "l"(__double_as_longlong(v)), "r"(remote_addr(bar, rank)) : "memory");
}

__device__ __forceinline__ bool wait_column(uint64_t *bar, long long t0)
{
    for (;;) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(tc::smem_addr(bar)), "r"(0u) : "memory");
        if (ok) return true;
        if (clock64() - t0 > kFactorWaitCycles) return false;
    }
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// v > 0, NaN excluded (on the bits: an FP64 compare would hold the FP64 unit).
__device__ __forceinline__ bool positive(double v)
{
    return (unsigned long long)__double_as_longlong(v) - 1ull < 0x7FF0000000000000ull;
}

// Shared memory of a CTA for a factor of at most n_ctas x 16 rows: columns U[k][j], the own rows'
// a_jk as they are updated and the earlier CTAs' a_jk as they were when column k was taken;
// 1 / a_kk, a_kk, the scales 1 / sqrt(a_kk), and a barrier per column.
__host__ __device__ inline size_t factor_smem(int n_ctas)
{
    const size_t Dp = (size_t)kRows * n_ctas;
    return sizeof(double) * (Dp * Dp + 4 * Dp);
}

// Called by every thread of every CTA of the cluster (`n_ctas` CTAs; those past the last row
// only take part in the barriers). withhold: the first CTA sends nothing of column 0, so that the
// others' wait for it runs out on purpose (the test of this path).
__device__ __forceinline__ void factor_cluster(const double *C, double sigma2, int D, int n_ctas, double *L,
                                               float *Lt, uint32_t *status, double *smem, bool withhold)
{
    const int b = (int)cooperative_groups::this_cluster().block_rank();
    const int n_used = (D + kRows - 1) / kRows, Dp = kRows * n_ctas;
    double *U = smem, *s_d = U + (size_t)Dp * Dp, *s_v = s_d + Dp, *s_s = s_v + Dp;
    uint64_t *bar = reinterpret_cast<uint64_t *>(s_s + Dp);
    __shared__ int s_bad;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool live = b < n_used, worker = warp != 0;
    const int k0 = kRows * b, kend = min(k0 + kRows, D);   // own columns
    const int ri = lane & (kRows - 1), half = lane >> 4, row = k0 + ri;
    if (tid == 0) s_bad = 0;
    if (live)
        for (int k = tid; k < k0; k += kFactorThreads) {   // one message per earlier column and source
            tc::mbar_init(bar + k, 1);
            tc::mbar_init_fence();
            tc::mbar_expect_tx(bar + k, (uint32_t)(kRows * sizeof(double)) * (uint32_t)(b - k / kRows) + 16u);
        }
    cluster_barrier();   // every barrier is ready before a message can arrive
    if (live) {
        for (int idx = tid; idx < kRows * (k0 + kRows); idx += kFactorThreads) {
            const int r = k0 + idx % kRows, c = idx / kRows;
            U[(size_t)c * Dp + r] = r < D && c <= r ? sigma2 * C[(size_t)r * D + c] : 0.0;
        }
        __syncthreads();
        // The column pairs dealt to warps w = 0 .. W - 1. publish: column k of the own rows to the
        // later CTAs, by the warp that holds its pair.
        auto publish = [&](int k, int w, int W) {
            if ((k >> 1) % W != w || half != (k & 1)) return;
            const double *at = U + (size_t)k * Dp + row, u = *at;
            for (int r = b + 1; r < n_used; ++r) send_double(at, bar + k, r, u);
        };
        // a_ij -= t_i a_jk for the own rows and the columns after k, but not for the next pivot
        // of the own columns (warp 0's). q: the first pair of this warp with a column after k.
        auto apply = [&](int k, int w, int W) {
            const double *Uk = U + (size_t)k * Dp;
            const double t = Uk[row] * s_d[k];
            const int first = (k + 1) >> 1;
            int q = first + (w - first % W + W) % W;
#pragma unroll 2
            for (; 2 * q < k0 + kRows; q += W) {
                const int j = 2 * q + half;
                double *at = U + (size_t)j * Dp + row;
                const double x = fma(-t, Uk[j], *at);
                if (j > k && !(k >= k0 && j == k + 1 && row == j)) *at = x;
            }
        };
        if (!withhold) publish(0, warp, kWarps);
        __syncthreads();
        bool late = false;
        for (int k = 0; k < k0; ++k) {   // columns of the earlier CTAs
            if (!late && !wait_column(bar + k, clock64())) {
                late = true;
                atomicOr(status, DEV_ERR_TIMEOUT);
            }
            apply(k, warp, kWarps);
            publish(k + 1, warp, kWarps);
            __syncthreads();
        }
        double v = 0.0, d = 0.0;   // the current pivot and its reciprocal
        auto pivot = [&](int k, double x) {
            v = x;
            if (!positive(v)) {
                v = 1.0;
                if (lane == 0) s_bad = 1;
            }
            d = recip_newton(v);
            if (lane == 0) {
                s_d[k] = d;
                s_v[k] = v;
            }
        };
        if (!worker) pivot(k0, U[(size_t)k0 * Dp + k0]);
        __syncthreads();
        for (int k = k0; k < kend; ++k) {   // own columns
            if (worker) {
                if (k + 1 < kend) {
                    apply(k, warp - 1, kWorkers);
                    publish(k + 1, warp - 1, kWorkers);
                }
            } else {
                const double dk = d, vk = v;
                double x = 0.0;
                if (k + 1 < kend) {
                    const double u = U[(size_t)k * Dp + k + 1];
                    x = fma(-(u * dk), u, U[(size_t)(k + 1) * Dp + k + 1]);
                }
                if (lane > b && lane < n_used && !(withhold && k == 0)) {   // while the chain above runs
                    send_double(s_d + k, bar + k, lane, dk);
                    send_double(s_v + k, bar + k, lane, vk);
                }
                if (k + 1 < kend) pivot(k + 1, x);
            }
            __syncthreads();
        }
        for (int k = tid; k < kend; k += kFactorThreads) s_s[k] = rsqrt_newton(s_v[k]);
        __syncthreads();
        const int rows = kend - k0;
        for (int idx = tid; idx < rows * D; idx += kFactorThreads) {
            const int r = k0 + idx / D, c = idx % D;
            const double l = c < r ? U[(size_t)c * Dp + r] * s_s[c] : (c == r ? s_v[r] * s_s[r] : 0.0);
            L[(size_t)r * D + c] = l;
        }
        for (int idx = tid; idx < rows * D; idx += kFactorThreads) {   // consecutive rows per column
            const int c = idx / rows, r = k0 + idx % rows;
            const double l = c < r ? U[(size_t)c * Dp + r] * s_s[c] : (c == r ? s_v[r] * s_s[r] : 0.0);
            Lt[(size_t)c * D + r] = (float)l;
        }
        if (tid == 0 && s_bad && !late) atomicOr(status, DEV_ERR_NOT_PD);
        if (late) {   // what the others still send arrives here: awaited too, with one limit for all
            const long long t0 = clock64();
            for (int k = 0; k < k0; ++k) wait_column(bar + k, t0);
        }
    }
    cluster_barrier();   // no CTA leaves while a message to it or from it may be under way
}

__global__ void __launch_bounds__(kFactorThreads)
k_factor(const double *C, double sigma2, const double *sigma_dev, int D, double *L,
         float *Lt, uint32_t *status, int withhold)
{
    after_previous();
    extern __shared__ __align__(16) double sm[];
    if (sigma_dev != nullptr) sigma2 = sigma_dev[0] * sigma_dev[0];   // the step size kept on the device
    factor_cluster(C, sigma2, D, (int)gridDim.x, L, Lt, status, sm, withhold != 0);
}

// The factors of every query of a batch, one cluster per query.
__global__ void __launch_bounds__(kFactorThreads)
k_batch_factor_cluster(const BatchQueryDev *__restrict__ qd, int n_ctas)
{
    extern __shared__ __align__(16) double sm[];
    const BatchQueryDev &q = qd[blockIdx.x / n_ctas];
    factor_cluster(q.C, q.sigma2, q.D, n_ctas, q.L, q.Lt, q.status, sm, false);
}

std::atomic<int> g_withhold_factor{0};   // test hook

struct ClusterLaunch {
    cudaLaunchAttribute attr[2] = {};
    cudaLaunchConfig_t cfg{};
    ClusterLaunch(int blocks, int n_ctas, cudaStream_t st, bool chained)
    {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = n_ctas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // k_factor: chain_launch.cuh
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(kFactorThreads);
        cfg.dynamicSmemBytes = factor_smem(n_ctas);
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = chained ? 2 : 1;
    }
};

}  // namespace

int factor_configure()
{
    CP_CUDA(cudaFuncSetAttribute(k_factor, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)factor_smem(kMaxCtas)));
    CP_CUDA(cudaFuncSetAttribute(k_batch_factor_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)factor_smem(kMaxCtas)));
    return CP_OK;
}

int launch_factor(const double *C, double sigma2, const double *sigma_dev, int D, double *L,
                  float *Lt_f, uint32_t *status, cudaStream_t st)
{
    const int n_ctas = (D + kRows - 1) / kRows;
    const ClusterLaunch l(n_ctas, n_ctas, st, true);
    CP_CUDA(cudaLaunchKernelEx(&l.cfg, k_factor, C, sigma2, sigma_dev, D, L, Lt_f, status, g_withhold_factor.load()));
    CP_LAUNCHED("k_factor");
    return CP_OK;
}

int batch_factor_clusters(int max_D, int *count)
{
    const int n_ctas = (max_D + kRows - 1) / kRows;
    const ClusterLaunch l(n_ctas, n_ctas, nullptr, false);   // the grid a whole number of clusters
    CP_CUDA(cudaOccupancyMaxActiveClusters(count, k_batch_factor_cluster, &l.cfg));
    return CP_OK;
}

int launch_batch_factor_cluster(const BatchQueryDev *qd, int nq, int max_D, cudaStream_t st)
{
    const int n_ctas = (max_D + kRows - 1) / kRows;
    const ClusterLaunch l(nq * n_ctas, n_ctas, st, false);
    CP_CUDA(cudaLaunchKernelEx(&l.cfg, k_batch_factor_cluster, qd, n_ctas));
    CP_LAUNCHED("k_batch_factor_cluster");
    return CP_OK;
}

}  // namespace cp

extern "C" void cp_debug_withhold_factor(int32_t on) { cp::g_withhold_factor.store(on != 0); }
