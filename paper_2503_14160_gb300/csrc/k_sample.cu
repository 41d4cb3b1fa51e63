// Algorithm 1 step (1): xi_i ~ N(mu, sigma^2 C) (arXiv 2503.14160, Sec. 4.1).
//   k_batch_factor  L L^T = sigma^2 C of many queries, FP64 right-looking Cholesky (L D L^T form),
//             one CTA per query, D <= 128 (one query or few: a cluster each, k_factor.cu)
//   k_sample  z_i from Philox4x32-10 (Salmon et al., SC'11) + Box-Muller, xi_i = mu + L z_i
// The counter of candidate i, block j, iteration t, query q is (j, i, t, q); the key is
// the 64-bit seed split into two words. Block j gives the normals z[4j..4j+3].
#include <algorithm>

#include "chain_launch.cuh"
#include "cp_internal.cuh"
#include "fp64_chain.cuh"
#include "philox.cuh"

namespace cp {
namespace {

__global__ void k_philox(const uint4 *__restrict__ ctr, uint32_t k0, uint32_t k1, int64_t n,
                         uint4 *out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = philox4x32_10(ctr[i], k0, k1);
}

constexpr int kFactorThreads = 1024;
constexpr int kFactorMaxD = 4 * CP_MAX_WAYPOINTS;

// One CTA, right-looking Cholesky of A = sigma^2 C in shared memory (row stride D + 1) in
// the unscaled (L D L^T) form: step k takes t_i = a_ik / a_kk for the rows below the pivot,
// then a_ij -= t_i a_jk over the trailing lower triangle, one FMA per entry and every lane
// busy. The next pivot's reciprocal is the critical chain of every column; the FP64 pipe is
// narrow, so that chain runs alone on one scheduler: warps are dealt to the SM's four
// schedulers round robin, warp 0 computes a_{k+1,k+1} and its reciprocal (double
// buffered), and the bulk update runs on the warps of the other three schedulers. At the
// end column k holds a_ik = l_ik sqrt(a_kk), so l_ik = a_ik / sqrt(a_kk) with the D square
// roots taken together. Outputs L (double, row-major, upper part zero) and its FP32
// transpose Lt[c][r] = L[r][c] for the sampler. A pivot that is not positive raises
// DEV_ERR_NOT_PD (and is replaced by 1 so that the kernel finishes).
__device__ __forceinline__ void factor_body(const double *__restrict__ C, double sigma2, int D, double *L,
                                            float *Lt, uint32_t *status, double *A)
{
    __shared__ double s_d[2];
    __shared__ double s_t[kFactorMaxD];
    __shared__ int bad;
    const int ld = D + 1;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const bool worker = (warp & 3) != 0;
    const int wtid = ((warp >> 2) * 3 + (warp & 3) - 1) * 32 + lane;   // 0 .. 3/4 blockDim - 1
    const int wcount = (int)blockDim.x / 4 * 3;
    for (int idx = tid; idx < D * D; idx += blockDim.x) {
        const int r = idx / D, c = idx - r * D;
        if (c <= r) A[r * ld + c] = sigma2 * C[idx];
    }
    __syncthreads();
    if (tid == 0) {
        bad = 0;
        double a = A[0];
        if (!(a > 0.0)) {
            bad = 1;
            a = 1.0;
            A[0] = a;
        }
        s_d[0] = recip_newton(a);
    }
    __syncthreads();
    for (int k = 0; k + 1 < D; ++k) {
        const int T = D - k - 1;
        const double d = s_d[k & 1];
        if (worker)
            for (int i = wtid; i < T; i += wcount) s_t[i] = A[(k + 1 + i) * ld + k] * d;
        __syncthreads();
        if (worker) {
            const int E = T * (T + 1) / 2;
            for (int e = wtid + 1; e < E; e += wcount) {   // entry 0 is the pivot
                int ii, jj;
                tri_index(e, ii, jj);
                const int i = k + 1 + ii, j = k + 1 + jj;
                A[i * ld + j] = fma(-s_t[ii], A[j * ld + k], A[i * ld + j]);
            }
        } else if (tid == 0) {
            const int i = k + 1;
            double v = fma(-(A[i * ld + k] * d), A[i * ld + k], A[i * ld + i]);
            if (!(v > 0.0)) {
                bad = 1;
                v = 1.0;
            }
            A[i * ld + i] = v;
            s_d[(k + 1) & 1] = recip_newton(v);
        }
        __syncthreads();
    }
    for (int k = tid; k < D; k += blockDim.x) s_t[k] = rsqrt_newton(A[k * ld + k]);
    __syncthreads();
    for (int idx = tid; idx < D * D; idx += blockDim.x) {
        const int r = idx / D, c = idx - r * D;
        const double l = c <= r ? A[r * ld + c] * s_t[c] : 0.0;
        L[idx] = l;
        Lt[c * D + r] = (float)l;
    }
    __syncthreads();
    if (tid == 0 && bad) atomicOr(status, DEV_ERR_NOT_PD);
}

// The factors of every query of a batch, one CTA per query.
__global__ void __launch_bounds__(kFactorThreads) k_batch_factor(const BatchQueryDev *__restrict__ qd)
{
    extern __shared__ double A[];
    const BatchQueryDev &q = qd[blockIdx.x];
    factor_body(q.C, q.sigma2, q.D, q.L, q.Lt, q.status, A);
}

// The sampler's tile: a warp draws 2 Q candidates, its lower half the first Q and its upper half
// the others; lane l of a half holds rows l, l + 16, .. of L z for all of its Q. Both operands of
// an FMA come from shared memory, which delivers 128 bytes per cycle to the SM, a word broadcast to
// 32 lanes like 32 words: with one row and eight candidates per lane, nine words per eight FMAs,
// that bounded the kernel. With eight rows and eight candidates it is 16 per 64.
// N = 65536, D = 128: 104 us in the former shape, 90 with the mean added in FP32, 54 now.
constexpr int kSampleWarps = 8;
constexpr int kSampleThreads = 32 * kSampleWarps;
constexpr int kRowBlock = 16;                              // rows of a block, columns of a segment
constexpr int kMaxBlocks = 4 * CP_MAX_WAYPOINTS / kRowBlock;   // 8

// Row blocks that the sampler computes for dimension D: an even number (the forms compiled).
__host__ __device__ constexpr int sample_blocks(int D) { return (D + 2 * kRowBlock - 1) / (2 * kRowBlock) * 2; }

// Floats of the staged factor: column c of segment k = c / 16 from row 16 k on (the rows above
// hold zeros of L).
__host__ __device__ constexpr int staged_floats(int nb) { return kRowBlock * kRowBlock * nb * (nb + 1) / 2; }

// Shared memory of the sampler: the staged L^T (FP32), the mean's rows as MeanRow and per warp the
// normals of its 2 Q candidates ([D][2 Q], candidate fastest).
size_t sample_smem(int K, int Q)
{
    const int D = 4 * K, nb = sample_blocks(D);
    return sizeof(float) * ((size_t)staged_floats(nb) + 4 * D + (size_t)kSampleWarps * 2 * Q * D);
}

// A row of the mean for sum_rounded: m = hi + lo + r, |r| <= 2^-48 |m| + 2^-150 < slack / 2.
struct __align__(16) MeanRow {
    float hi, lo, slack, pad;
};

__device__ __forceinline__ MeanRow mean_row(double m)
{
    const float hi = (float)m;
    return {hi, (float)(m - (double)hi), fmaxf(fabsf(hi) * 0x1p-46f, 0x1p-140f), 0.f};
}

// float(m + a), the sum rounded to FP64 and then to FP32, in FP32: s + e = hi + a exactly (Knuth's
// two-sum), t = e + lo, and the true sum lies in s + t -+ d, d covering the roundings of t, lo, the
// bracket's own and the FP64 sum's (2^-53 |sum|, below 2^-22 |t| wherever t reaches half an FP32
// step). Rounding is monotone, so where both ends round to one float that is the result; else
// (a sum within 2^-22 of a tie, infinities, NaN) false.
__device__ __forceinline__ bool sum_rounded(const MeanRow &m, float a, float &x)
{
    const float s = __fadd_rn(m.hi, a), b = __fadd_rn(s, -m.hi);
    const float e = __fadd_rn(__fadd_rn(m.hi, -__fadd_rn(s, -b)), __fadd_rn(a, -b));
    const float t = __fadd_rn(e, m.lo), d = __fmaf_rn(fabsf(t), 0x1p-22f, m.slack);
    x = __fadd_rn(s, __fadd_rn(t, d));
    return x == __fadd_rn(s, __fadd_rn(t, -d));
}

__device__ __noinline__ float sum_fp64(const double *mu, int r, float a) { return (float)(mu[r] + (double)a); }

// The normals of candidates g .. g + 2 Q - 1 (Philox counter (j, i, iter, query) for z[4j..4j+3],
// spread over the lanes) into the warp's buffer.
template <int Q>
__device__ __forceinline__ void draw_normals(float *sZ, int K, uint32_t k0, uint32_t k1, uint32_t iter, uint32_t query,
                                             int g, int i_end, int lane)
{
    for (int pq = lane; pq < 2 * Q * K; pq += 32) {
        const int cnd = pq % (2 * Q), j = pq / (2 * Q);
        const int i = g + cnd;
        float z0 = 0.f, z1 = 0.f, z2 = 0.f, z3 = 0.f;
        if (i < i_end) {
            const uint4 x = philox4x32_10(make_uint4((uint32_t)j, (uint32_t)i, iter, query), k0, k1);
            box_muller(x.x, x.y, z0, z1);
            box_muller(x.z, x.w, z2, z3);
        }
        sZ[(4 * j + 0) * 2 * Q + cnd] = z0;
        sZ[(4 * j + 1) * 2 * Q + cnd] = z1;
        sZ[(4 * j + 2) * 2 * Q + cnd] = z2;
        sZ[(4 * j + 3) * 2 * Q + cnd] = z3;
    }
    __syncwarp();
}

// xi of the warp's candidates: acc = sum_c L[r][c] z[c] over ascending c with one FMA per term, then
// xi_r = mu_r + acc (added in FP64, rounded once to FP32: by sum_rounded, as the conversion, the
// addition and the conversion back hold the scheduler's FP64 unit for 205 cycles per 32 entries).
// Columns past the last one of a row's block hold zeros of L for every row of the block and are
// skipped; adding 0 z leaves a nonzero sum unchanged, so each row equals the full D-term sum.
template <int Q, int NB>
__device__ __forceinline__ void multiply_rows(const double *mu, const float *sL, const MeanRow *sM,
                                              const float *sZ, int D, float *xi, int g, int i_end, int lane)
{
    const int row = lane & (kRowBlock - 1), half = lane >> 4;
    float acc[NB][Q];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[b][q] = 0.f;
    const float *l = sL + row, *zc = sZ + Q * half;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const int n = min(D - kRowBlock * k, kRowBlock);   // columns of the segment (none: <= 0)
#pragma unroll 2
        for (int c = 0; c < n; ++c) {
            float z[Q];
#pragma unroll
            for (int q = 0; q < Q; q += 2) {
                const float2 v = *reinterpret_cast<const float2 *>(zc + q);
                z[q] = v.x;
                z[q + 1] = v.y;
            }
#pragma unroll
            for (int b = k; b < NB; ++b) {
                const float lv = l[kRowBlock * (b - k)];
#pragma unroll
                for (int q = 0; q < Q; ++q) acc[b][q] = fmaf(lv, z[q], acc[b][q]);
            }
            l += kRowBlock * (NB - k);
            zc += 2 * Q;
        }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int r = kRowBlock * b + row;
        if (r < D) {
            const MeanRow m = sM[r];
            bool ok = true;
            float x[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) ok = sum_rounded(m, acc[b][q], x[q]) && ok;
            if (!ok)
#pragma unroll
                for (int q = 0; q < Q; ++q) x[q] = sum_fp64(mu, r, acc[b][q]);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int i = g + Q * half + q;
                if (i < i_end) xi[(size_t)i * D + r] = x[q];
            }
        }
    }
    __syncwarp();
}

// Warp w draws the groups of 2 Q candidates from g0 + 2 Q w on, g_stride apart, below i_end.
// kWait: the mean and the factor come from the launch before (its end is awaited after
// the first group's normals, which need neither).
template <int Q, bool kWait>
__device__ __forceinline__ void sample_body(const double *mu, const float *Lt, int K,
                                            uint32_t k0, uint32_t k1, uint32_t iter, uint32_t query,
                                            float *xi, int g0, int g_stride, int i_end, float *sm)
{
    const int D = 4 * K, nb = sample_blocks(D), rows = kRowBlock * nb;
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *sL = sm;
    MeanRow *sM = reinterpret_cast<MeanRow *>(sm + staged_floats(nb));
    float *sZ = sm + staged_floats(nb) + 4 * D + wib * 2 * Q * D;
    const int first = g0 + 2 * Q * wib;
    draw_normals<Q>(sZ, K, k0, k1, iter, query, first, i_end, lane);
    if (kWait) after_previous();
    // 16-byte pieces of the columns, all in flight together (rows past D: zeros)
    for (int k = 0, at = 0; k < nb; ++k) {
        const int top = kRowBlock * k, pieces = (rows - top) / 4;
        for (int e = threadIdx.x; e < min(kRowBlock, D - top) * pieces; e += kSampleThreads) {
            const int c = top + e / pieces, r = top + 4 * (e % pieces);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::
                         "r"((uint32_t)__cvta_generic_to_shared(sL + at + 4 * e)),
                         "l"(Lt + (r < D ? c * D + r : 0)), "r"(r < D ? 16 : 0) : "memory");
        }
        at += kRowBlock * 4 * pieces;
    }
    for (int r = threadIdx.x; r < D; r += blockDim.x) sM[r] = mean_row(mu[r]);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int g = first; g < i_end; g += g_stride) {
        if (g != first) draw_normals<Q>(sZ, K, k0, k1, iter, query, g, i_end, lane);
        switch (nb) {
        case 2: multiply_rows<Q, 2>(mu, sL, sM, sZ, D, xi, g, i_end, lane); break;
        case 4: multiply_rows<Q, 4>(mu, sL, sM, sZ, D, xi, g, i_end, lane); break;
        case 6: multiply_rows<Q, 6>(mu, sL, sM, sZ, D, xi, g, i_end, lane); break;
        default: multiply_rows<Q, kMaxBlocks>(mu, sL, sM, sZ, D, xi, g, i_end, lane); break;
        }
    }
}

template <int Q>
__global__ void __launch_bounds__(kSampleThreads, 2)
k_sample(const double *mu, const float *Lt, int N, int K,
         uint32_t k0, uint32_t k1, uint32_t iter, uint32_t query, float *xi)
{
    extern __shared__ __align__(16) float sm[];
    const int per_block = kSampleWarps * 2 * Q;
    sample_body<Q, true>(mu, Lt, K, k0, k1, iter, query, xi, blockIdx.x * per_block, gridDim.x * per_block, N, sm);
}

constexpr int kBatchQ = 8;

// Every query's draw in one launch: block b of query q takes the kBatchSampleCands
// candidates from b kBatchSampleCands, each warp several groups in turn (the
// block stages the query's factor once for all of them). A candidate's normals and
// arithmetic do not depend on which warp draws it, so each query's xi equals its plain draw.
__global__ void __launch_bounds__(kSampleThreads, 2)
k_batch_sample(const BatchQueryDev *__restrict__ qd, const int2 *__restrict__ tab, uint32_t iter)
{
    extern __shared__ __align__(16) float sm[];
    const int2 e = tab[blockIdx.x];
    const BatchQueryDev &q = qd[e.x];
    const int b = e.y * kBatchSampleCands;
    static_assert(kBatchSampleCands % (kSampleWarps * 2 * kBatchQ) == 0, "whole groups of candidates per warp");
    sample_body<kBatchQ, false>(q.mu, q.Lt, q.K, q.seed_lo, q.seed_hi, iter, q.query, q.xi, b,
                                kSampleWarps * 2 * kBatchQ, min(q.N, b + kBatchSampleCands), sm);
}

}  // namespace

int launch_philox(const uint32_t *ctr, uint32_t k0, uint32_t k1, int64_t n, uint32_t *out,
                  cudaStream_t st)
{
    if (n == 0) return CP_OK;
    const int threads = 256;
    const int64_t blocks = (n + threads - 1) / threads;
    k_philox<<<(unsigned)blocks, threads, 0, st>>>((const uint4 *)ctr, k0, k1, n, (uint4 *)out);
    CP_LAUNCHED("k_philox");
    return CP_OK;
}

int sample_configure()
{
    const int smem = (int)sample_smem(CP_MAX_WAYPOINTS, 8);
    CP_CUDA(cudaFuncSetAttribute(k_sample<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CP_CUDA(cudaFuncSetAttribute(k_sample<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CP_CUDA(cudaFuncSetAttribute(k_sample<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CP_CUDA(cudaFuncSetAttribute(k_batch_sample, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const int Dm = 4 * CP_MAX_WAYPOINTS;
    CP_CUDA(cudaFuncSetAttribute(k_batch_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(double) * Dm * (Dm + 1))));
    return CP_OK;
}

// One cluster per query while they fill the device at most kClusterWaves times, else one CTA per
// query: at D = 128 a cluster takes about 80 us and holds eight SMs, a CTA 198 us and one SM
// (the same bits), so two waves of clusters are still the faster form and three are not.
constexpr int kClusterWaves = 2;

int launch_batch_factor(const BatchQueryDev *qd, int nq, int max_D, cudaStream_t st)
{
    int fit = 0;
    const int rc = batch_factor_clusters(max_D, &fit);
    if (rc != CP_OK) return rc;
    if (nq <= kClusterWaves * fit) return launch_batch_factor_cluster(qd, nq, max_D, st);
    const size_t smem = sizeof(double) * (size_t)max_D * (max_D + 1);
    k_batch_factor<<<nq, kFactorThreads, smem, st>>>(qd);
    CP_LAUNCHED("k_batch_factor");
    return CP_OK;
}

int launch_batch_sample(const BatchQueryDev *qd, const int2 *tab, int blocks, int max_K, uint32_t iter,
                        cudaStream_t st)
{
    if (blocks == 0) return CP_OK;
    k_batch_sample<<<blocks, kSampleThreads, sample_smem(max_K, kBatchQ), st>>>(qd, tab, iter);
    CP_LAUNCHED("k_batch_sample");
    return CP_OK;
}

// Candidates per warp: the fewest of 4, 8 and 16 whose blocks of eight warps all have an SM to
// themselves, else 16. More per warp take fewer shared-memory words per FMA, fewer make more warps
// and a shorter chain of one draw and one product. us with 4, 8 and 16 (former kernel):
//   N = 4096, D = 128: 8.0, 9.2, 14.4 (23.6);   N = 8192, D = 128: 11.3, 10.0, 14.6 (23.6);
//   N = 16384, D = 128: 20.0, 16.2, 15.6 (31.2);   N = 256, D = 32: 2.9, 3.1, 3.6 (4.1).
template <int Q>
int launch_sample_form(int sms, const double *mu, const float *Lt_f, int N, int K, uint64_t seed, uint32_t iter,
                       uint32_t query, float *xi, cudaStream_t st)
{
    int per_sm = 0;
    const size_t smem = sample_smem(K, Q);
    CP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample<Q>, kSampleThreads, smem));
    if (per_sm < 1) per_sm = 1;
    const int per_block = kSampleWarps * 2 * Q, blocks = std::min((N + per_block - 1) / per_block, sms * per_sm);
    launch_chained(k_sample<Q>, blocks, kSampleThreads, smem, st, mu, Lt_f, N, K, (uint32_t)seed,
                   (uint32_t)(seed >> 32), iter, query, xi);
    CP_LAUNCHED("k_sample");
    return CP_OK;
}

int launch_sample(const double *mu, const float *Lt_f, int N, int K, uint64_t seed,
                  uint32_t iter, uint32_t query, float *xi, cudaStream_t st)
{
    int dev = 0, sms = 0;
    CP_CUDA(cudaGetDevice(&dev));
    CP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (N <= sms * kSampleWarps * 4) return launch_sample_form<2>(sms, mu, Lt_f, N, K, seed, iter, query, xi, st);
    if (N <= sms * kSampleWarps * 8) return launch_sample_form<4>(sms, mu, Lt_f, N, K, seed, iter, query, xi, st);
    return launch_sample_form<8>(sms, mu, Lt_f, N, K, seed, iter, query, xi, st);
}

}  // namespace cp
