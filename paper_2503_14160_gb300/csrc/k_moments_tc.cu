// Weighted mean and covariance of many elites (Algorithm 1 steps (5)-(6); arXiv 2503.14160, Sec.
// 4.1) as exact integer products on the tensor cores.
//
// What bounds it. S2 = sum_j w_j y_j y_j^T over nu elites (y_j = x_(j) - x_(1)) is nu D^2 / 2 FP64
// FMAs, and this part issues one FP64 warp instruction per scheduler in 64 cycles: 544 us for
// nu = 32768, D = 128, with 34 us more for y and w y in FP64. The split below keeps FP64's
// accuracy and runs on the tensor cores' BF16 rate (Ootomo, Ozaki and Yokota's integer form of
// the Ozaki scheme, "DGEMM on integer matrix multiplication unit", 2024, with BF16 products that
// FP32 accumulates exactly):
//   z_j = sqrt(w_j) y_j, so S2 = Z^T Z. Per column c the deviations are 55-bit integers
//   Y = y 2^(54 - ey_c), |y| < 2^ey_c over the elites (k_moments_range): the difference of two
//   floats as integers, with wrap-around subtraction, so no FP64 instruction is issued. sqrt(w_j) is a
//   63-bit integer, and Z = (Y W) >> 63, rounded, has 54 bits and a sign.
//   Z = sum_s d_s 2^(8 (6 - s)), s = 0 .. 6, digits d_s in [-128, 127], exact in BF16.
//   S2 = sum over digit pairs of products of integers below 2^14. Pairs of equal weight s + t = l
//   share an FP32 accumulator; with at most six pairs (98304 per elite) and 128 elites its
//   integers stay below 2^24, so FP32 accumulates them exactly. Levels l = 0 .. 7 are kept (34
//   products); what is left out is below 2^-62 of the largest z^2 per elite.
//   Every 128 elites the accumulators are added as 64-bit integers, and so are the CTAs' sums:
//   the result does not depend on the split, and the only roundings are those of Z (2^-55 of the
//   column's largest deviation times the largest weight's root) and of the final FP64 value.
// S1 = sum_j w_j y_j takes the same integers Y times a 63-bit w_j.
//
// A CTA takes 64 columns of S2 (all 128 rows) over a range of elites, 32 at a time: 1024 threads
// turn one column of four elites each into digits in shared memory (K-major core matrices) while
// the tensor cores work on the stage before, one thread issues the 68 MMAs of 128 x 64 x 16, and
// the eight levels fill the 512 columns of tensor memory. nu = 32768, D = 128: 84 us, with 9 us for
// the columns' ranges and 11 us for the final sums; cp_update of 65536 candidates 241 us, and 740 us
// with the FP64 form. A plan's and a batch's updates keep the FP64 sums (see run_update).
#include "chain_launch.cuh"
#include "cp_internal.cuh"
#include "tcgen05.cuh"

namespace cp {
namespace {

constexpr int kTcThreads = 1024;
constexpr int kTcRows = 128;            // rows of S2 (D <= 128), the MMA's M
constexpr int kTcCols = 64;             // columns of S2 per CTA, the MMA's N
constexpr int kStage = 32;              // elites per stage (two K steps of 16)
constexpr int kPer = kStage * kTcRows / kTcThreads;                // elites of a thread per stage: 4
constexpr int kAcc = kTcRows * kTcCols / kTcThreads;               // entries of a thread: 8
constexpr int kEpoch = 4;               // stages per accumulation: 128 elites
constexpr int kDigits = 7, kLevels = 8;
constexpr uint32_t kLbo = 128, kSbo = kStage / 8 * 128;            // core-matrix offsets, bytes
constexpr int kSliceBytes = kTcRows * kStage * 2;                  // one digit of a stage
constexpr int kStageBytes = kDigits * kSliceBytes;
constexpr size_t kTcSmem = 2 * (size_t)kStageBytes;
constexpr uint32_t kTmemCols = kLevels * kTcCols;                  // 512
constexpr long long kTcWaitCycles = 2000000000ll;                  // about one second
constexpr int kFrac = 54;               // bits of Y below the column's bound

// Exponent bound of a column: |y| < 2^ey for the largest |y| whose float has these bits.
__device__ __forceinline__ int bound_exponent(uint32_t bits) { return max((int)(bits >> 23), 1) - 126; }

__device__ __forceinline__ bool column_finite(uint32_t bits) { return bits < 0x7F800000u; }

// x 2^(54 - ey) modulo 2^64 (bits below the last place cut); wrap-around is harmless, as only
// differences below 2^55 in magnitude are formed from it.
__device__ __forceinline__ long long fixed_of(float x, int ey)
{
    const uint32_t b = __float_as_uint(x), e = (b >> 23) & 255u;
    const unsigned long long mant = (unsigned long long)((b & 0x7FFFFFu) | (e != 0u ? 0x800000u : 0u));
    const int s = max((int)e, 1) - 150 + kFrac - ey;
    unsigned long long left, right;
    asm("shl.b64 %0, %1, %2;" : "=l"(left) : "l"(mant), "r"(max(s, 0)));     // counts above 63 give 0
    asm("shr.u64 %0, %1, %2;" : "=l"(right) : "l"(mant), "r"(max(-s, 0)));
    const long long v = (long long)(s >= 0 ? left : right);
    return (b >> 31) ? -v : v;
}

// (Y W) >> (63 + drop) rounded, for |Y| < 2^55 and 0 <= W < 2^63.
__device__ __forceinline__ long long scale63(long long Y, long long W, int drop = 0)
{
    return (__mul64hi((long long)((unsigned long long)Y << 5), W) + (8ll << drop)) >> (4 + drop);
}

// Bits dropped from the terms of S1, so that their sum, below 2^(54 - ew) as the weights sum to
// one, stays below 2^61.
__device__ __forceinline__ int mean_drop(int ew) { return max(0, -ew - 7); }

__device__ __forceinline__ void range_body(const MomentsTc &a, int block, int blocks)
{
    __shared__ uint32_t s_max[kTcRows];
    const int c = threadIdx.x & (kTcRows - 1), g = threadIdx.x / kTcRows, G = blockDim.x / kTcRows;
    if (threadIdx.x < kTcRows) s_max[threadIdx.x] = 0u;
    __syncthreads();
    if (c < a.D) {
        const float x0 = a.elites[c];
        uint32_t m = 0u;
#pragma unroll 8
        for (int j = block * G + g; j < a.nu; j += blocks * G)
            m = max(m, __float_as_uint(fabsf(a.elites[(size_t)j * a.D + c] - x0)));
        atomicMax(&s_max[c], m);
    }
    __syncthreads();
    if (threadIdx.x < a.D) atomicMax(a.colmax + threadIdx.x, s_max[threadIdx.x]);
}

__device__ __forceinline__ void moments_tc_body(const MomentsTc &a, int tile, int part, int parts)
{
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    __shared__ __align__(8) uint64_t done[2];
    __shared__ uint32_t s_tmem;
    __shared__ unsigned long long s_s1[kTcRows];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *buf = tc_smem;
    const int stages = (a.nu + kStage - 1) / kStage;
    const int first = (int)((long long)part * stages / parts), last = (int)((long long)(part + 1) * stages / parts);
    const int n = last - first;
    if (tid == 0) {
        tc::mbar_init(&done[0], 1);
        tc::mbar_init(&done[1], 1);
        tc::mbar_init_fence();
    }
    if (warp == 0) tc::tmem_alloc(&s_tmem, kTmemCols);
    if (tid < kTcRows) s_s1[tid] = 0ull;
    for (int i = tid; i < 2 * kStageBytes / 16; i += kTcThreads)   // rows past D stay zero
        reinterpret_cast<uint4 *>(buf)[i] = make_uint4(0u, 0u, 0u, 0u);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = s_tmem;
    // this thread's column and its four elites of every stage
    const int c = tid & (kTcRows - 1), g = tid / kTcRows;
    const bool on = c < a.D, own = on && c / kTcCols == tile;
    const int ey = on ? bound_exponent(a.colmax[c]) : 0;
    const int drop = mean_drop(a.scale[1]);
    const long long X1 = on ? fixed_of(a.elites[c], ey) : 0;
    long long s1 = 0;
    long long hi[kAcc], lo[kAcc];
#pragma unroll
    for (int i = 0; i < kAcc; ++i) hi[i] = lo[i] = 0;
    bool late = false;
    // the stage's accumulators as integers: weights 2^24, 2^16, 2^8, 1 into hi (levels 0-3) and
    // lo (levels 4-7); warp w holds rows 32 (w mod 4) .. and columns 8 (w / 4) ..
    auto drain = [&]() {
        __syncwarp();
        const uint32_t at = tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(kAcc * (warp >> 2));
#pragma unroll
        for (int l = 0; l < kLevels; l += 2) {
            uint32_t v[2 * kAcc];
            tc::tmem_ld8_async(at + (uint32_t)(l * kTcCols), v);
            tc::tmem_ld8_async(at + (uint32_t)((l + 1) * kTcCols), v + kAcc);
            tc::tmem_ld_wait<2 * kAcc>(v);
#pragma unroll
            for (int i = 0; i < kAcc; ++i) {
                const long long p = (long long)__float2int_rn(__uint_as_float(v[i])) * (1 << 8 * (3 - (l & 3))) +
                                    (long long)__float2int_rn(__uint_as_float(v[kAcc + i])) * (1 << 8 * (2 - (l & 3)));
                if (l < 4) hi[i] += p;
                else lo[i] += p;
            }
        }
    };
    auto wait = [&](int i) {   // the MMAs of stage i have completed
        if (!late && !tc::mbar_wait(&done[i & 1], (uint32_t)(i >> 1) & 1u, kTcWaitCycles)) {
            late = true;
            if (a.status != nullptr) atomicOr(a.status, DEV_ERR_TIMEOUT);
        }
    };
    float x[kPer];   // this thread's elites of the next stage, loaded a stage ahead
    auto load = [&](int i) {
        const int j0 = (first + i) * kStage + kPer * g;
#pragma unroll
        for (int q = 0; q < kPer; ++q) x[q] = on && i < n && j0 + q < a.nu ? a.elites[(size_t)(j0 + q) * a.D + c] : 0.f;
    };
    load(0);
    for (int i = 0; i < n; ++i) {
        if (i >= 2) wait(i - 2);
        if (on) {
            unsigned char *dst = buf + (size_t)(i & 1) * kStageBytes + (uint32_t)(c >> 3) * kSbo +
                                 (uint32_t)(g >> 1) * kLbo + (uint32_t)(c & 7) * 16u + (uint32_t)(g & 1) * 8u;
            const int j0 = (first + i) * kStage + kPer * g;
            unsigned long long u[kPer];   // Z with every digit biased by 128
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const bool in = j0 + q < a.nu;
                const long long Y = in ? fixed_of(x[q], ey) - X1 : 0;
                const long long Z = in ? scale63(Y, a.W[j0 + q]) : 0;
                if (own && in) s1 += scale63(Y, a.Wf[j0 + q], drop);
                u[q] = (unsigned long long)Z + 0x0080808080808080ull;
            }
#pragma unroll
            for (int s = 0; s < kDigits; ++s) {
                const int byte = kDigits - 1 - s;   // digit s: bits 8 byte .. 8 byte + 7
                uint32_t w[kPer / 2];
#pragma unroll
                for (int q = 0; q < kPer / 2; ++q) {
                    const uint32_t p = byte < 4 ? (uint32_t)u[2 * q] : (uint32_t)(u[2 * q] >> 32);
                    const uint32_t r = byte < 4 ? (uint32_t)u[2 * q + 1] : (uint32_t)(u[2 * q + 1] >> 32);
                    // two biased digits b = 128 h + m in 16-bit lanes; as BF16 (128 + m) - (256 -
                    // 128 h) = b - 128, exact: 0x43mm is 128 + m, 0x4380 is 256 and 0x4300 is 128
                    const uint32_t x2 = __byte_perm(__byte_perm(p, r, (byte & 3) | ((4 + (byte & 3)) << 4)), 0u, 0x4140);
                    const uint32_t m2 = (x2 & 0x007F007Fu) | 0x43004300u, h2 = (x2 & 0x00800080u) ^ 0x43804380u;
                    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(w[q]) : "r"(m2), "r"(h2));
                }
                *reinterpret_cast<uint2 *>(dst + s * kSliceBytes) = make_uint2(w[0], w[1]);
            }
        }
        load(i + 1);
        tc::fence_async_smem();
        if (i > 0 && i % kEpoch == 0) {
            wait(i - 1);
            tc::fence_after_sync();
            drain();
            tc::fence_before_sync();
        }
        __syncthreads();
        if (tid == 0) {
            tc::fence_after_sync();
            const uint32_t base = tc::smem_addr(buf) + (uint32_t)(i & 1) * (uint32_t)kStageBytes;
            const uint32_t b0 = (uint32_t)(tile * kTcCols / 8) * kSbo;
            constexpr uint32_t idesc = tc::idesc_bf16(kTcRows, kTcCols);
#pragma unroll 1
            for (int ks = 0; ks < kStage / 16; ++ks) {
                const uint32_t o = base + 2 * kLbo * (uint32_t)ks;
                const bool fresh = i % kEpoch == 0 && ks == 0;
#pragma unroll
                for (int l = 0; l < kLevels; ++l) {
                    const int s0 = l < kDigits ? 0 : l - kDigits + 1;
#pragma unroll
                    for (int s = s0; s <= l - s0; ++s)
                        tc::mma_f16kind(tmem + (uint32_t)(l * kTcCols),
                                        tc::desc_kmajor(o + (uint32_t)(s * kSliceBytes), kLbo, kSbo),
                                        tc::desc_kmajor(o + (uint32_t)((l - s) * kSliceBytes) + b0, kLbo, kSbo), idesc,
                                        !(fresh && s == s0));
                }
            }
            tc::mma_commit(&done[i & 1]);
        }
    }
    if (n > 0) {
        wait(n - 1);
        tc::fence_after_sync();
        drain();
        tc::fence_before_sync();
    }
    if (own && s1 != 0) atomicAdd(&s_s1[c], (unsigned long long)s1);
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kTmemCols);
    // partials [part][tile][column][row]
    const int tiles = (a.D + kTcCols - 1) / kTcCols, row = 32 * (warp & 3) + lane;
    const size_t at = ((size_t)part * tiles + tile) * kTcCols;
#pragma unroll
    for (int i = 0; i < kAcc; ++i) {
        const size_t e = (at + kAcc * (warp >> 2) + i) * kTcRows + row;
        a.hi[e] = hi[i];
        a.lo[e] = lo[i];
    }
    if (tid < kTcRows && tid / kTcCols == tile) a.s1[(size_t)part * kTcRows + tid] = (long long)s_s1[tid];
}

constexpr int kCombGroups = 4;   // threads per row of the combine, each every fourth part

// Column `col` of C (rows r >= col, mirrored) and, from the diagonal, mu: integer sums over the
// parts, then FP64. A column with an infinite or NaN deviation has no scale: its entries take the
// plain FP64 sums over the elites, which carry the value through as the general form does.
__device__ __forceinline__ void combine_tc_body(const MomentsTc &a, int col, int parts)
{
    __shared__ long long s_hi[kCombGroups][kTcRows], s_lo[kCombGroups][kTcRows], s_s1[kCombGroups][kTcRows];
    __shared__ double s_mean[kTcRows];
    const int r = threadIdx.x & (kTcRows - 1), g = threadIdx.x / kTcRows;
    const int tiles = (a.D + kTcCols - 1) / kTcCols, tile = col / kTcCols;
    long long h = 0, l = 0, s = 0;
#pragma unroll 4
    for (int p = g; p < parts; p += kCombGroups) {
        const size_t e = (((size_t)p * tiles + tile) * kTcCols + (col - tile * kTcCols)) * kTcRows + r;
        h += a.hi[e];
        l += a.lo[e];
        s += a.s1[(size_t)p * kTcRows + r];
    }
    s_hi[g][r] = h;
    s_lo[g][r] = l;
    s_s1[g][r] = s;
    __syncthreads();
    const bool row = g == 0 && r < a.D;
    const uint32_t br = row ? a.colmax[r] : 0u, bc = a.colmax[col];
    const int es = a.scale[0], ew = a.scale[1];
    if (row) {
        for (int q = 1; q < kCombGroups; ++q) {
            h += s_hi[q][r];
            l += s_lo[q][r];
            s += s_s1[q][r];
        }
        double m = scalbn((double)s, bound_exponent(br) + ew + mean_drop(ew) - kFrac);
        if (!column_finite(br)) {
            m = 0.0;
            for (int j = 0; j < a.nu; ++j) m = fma(a.w[j], (double)a.elites[(size_t)j * a.D + r] - (double)a.elites[r], m);
        }
        s_mean[r] = m;
        if (r == col) a.mu[r] = (double)a.elites[r] + m;
    }
    __syncthreads();
    if (!row || r < col) return;
    double s2;
    if (column_finite(br) && column_finite(bc)) {
        h += l >> 32;                              // carry: h 2^32 + the low 32 bits of l
        const double q = fma((double)h, 4294967296.0, (double)(uint32_t)l);
        s2 = scalbn(q, bound_exponent(br) + bound_exponent(bc) + 2 * es + 40 - 2 * kFrac);
    } else {
        s2 = 0.0;
        for (int j = 0; j < a.nu; ++j) {
            const float *x = a.elites + (size_t)j * a.D;
            s2 = fma(a.w[j] * ((double)x[r] - (double)a.elites[r]), (double)x[col] - (double)a.elites[col], s2);
        }
    }
    double v = fma(-s_mean[r], s_mean[col], s2);
    if (r == col) v += a.eps;
    a.C[(size_t)r * a.D + col] = v;
    a.C[(size_t)col * a.D + r] = v;
}

__global__ void __launch_bounds__(256) k_moments_range(const MomentsTc a) { range_body(a, blockIdx.x, gridDim.x); }

__global__ void __launch_bounds__(kTcThreads, 1) k_moments_tc(const MomentsTc a)
{
    after_previous();
    moments_tc_body(a, blockIdx.y, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(kCombGroups *kTcRows) k_moments_tc_combine(const MomentsTc a, int parts)
{
    after_previous();
    combine_tc_body(a, blockIdx.x, parts);
}

// Integer weights: W = sqrt(w_j) 2^(63 - es) and Wf = w_j 2^(63 - ew), es and ew the exponents
// that bound the first (largest) weight's.
__global__ void k_moments_tc_weights(const double *__restrict__ w, int nu, long long *W, long long *Wf, int *scale)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int es = ilogb(sqrt(w[0])) + 1, ew = ilogb(w[0]) + 1;
    if (j == 0) {
        scale[0] = es;
        scale[1] = ew;
    }
    if (j >= nu) return;
    W[j] = (long long)scalbn(sqrt(w[j]), 63 - es);
    Wf[j] = (long long)scalbn(w[j], 63 - ew);
}

}  // namespace

// The tensor-core form is taken from nu D^2 = 2^23 on, where the FP64 form needs about 14 us of the
// whole GPU's FP64 units: there a cp_update takes 104 us against 124 (nu = 8192, D = 32) and 108
// against 114 (nu = 512, D = 128).
bool moments_use_tc(int nu, int D) { return (long long)nu * D * D >= (1ll << 23); }

static int moments_tc_stages(int nu) { return (nu + kStage - 1) / kStage; }
int moments_tc_tiles(int D) { return (D + kTcCols - 1) / kTcCols; }

int moments_tc_parts(int nu, int D, int num_sms)
{
    const int per = num_sms / moments_tc_tiles(D), stages = moments_tc_stages(nu);
    return stages < per ? stages : (per < 1 ? 1 : per);
}

size_t moments_tc_partial(int D, int parts) { return (size_t)parts * moments_tc_tiles(D) * kTcCols * kTcRows; }

int moments_tc_configure()
{
    CP_CUDA(cudaFuncSetAttribute(k_moments_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem));
    return CP_OK;
}

int launch_moments_tc_weights(const double *w, int nu, long long *W, long long *Wf, int *scale, cudaStream_t st)
{
    k_moments_tc_weights<<<(nu + 255) / 256, 256, 0, st>>>(w, nu, W, Wf, scale);
    CP_LAUNCHED("k_moments_tc_weights");
    return CP_OK;
}

int launch_moments_tc(const MomentsTc &a, int parts, int num_sms, cudaStream_t st)
{
    CP_CUDA(cudaMemsetAsync(a.colmax, 0, sizeof(uint32_t) * a.D, st));
    const int rows = (a.nu + 15) / 16;
    k_moments_range<<<rows < 4 * num_sms ? rows : 4 * num_sms, 256, 0, st>>>(a);
    CP_LAUNCHED("k_moments_range");
    launch_chained(k_moments_tc, dim3(parts, moments_tc_tiles(a.D)), kTcThreads, kTcSmem, st, a);
    CP_LAUNCHED("k_moments_tc");
    launch_chained(k_moments_tc_combine, a.D, kCombGroups * kTcRows, 0, st, a, parts);
    CP_LAUNCHED("k_moments_tc_combine");
    return CP_OK;
}

}  // namespace cp
