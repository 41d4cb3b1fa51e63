// Differentiable form of the cost and its adjoint (the smooth surrogate of Eq. path opt,
// arXiv 2503.14160 Sec. 4.1, used to polish candidates before trajectory optimisation):
//   J_s = sum_k |q(s_k) - q(s_{k-1})|^2 + w_c lambda_c sum_k sum_pairs beta softplus((m - sd)/beta)
//         + w_l sum_k sum_j (max(0, q - q_max)^2 + max(0, q_min - q)^2)
// q(s_k) is linear in the control points, so with r_k = dJ/dq(s_k) the gradient is
//   dJ/dP_g = sum_k [2 (q_k - q_{k-1}) (b_g(s_k) - b_g(s_{k-1})) + r_k^pen b_g(s_k)],
// r_k^pen chaining the softplus derivative through the signed-distance gradient and the
// kinematic Jacobian. One warp per candidate walks its checkpoints 32 at a time (one per
// lane), recomputing the forward pass (no tape); the per-control-point sums of a chunk are
// reduced over the lanes by a fixed butterfly into a per-warp accumulator, so results are
// deterministic.
//
// What bounds it: instruction issue, most of it in the pairs within the softplus range. An
// obstacle of a chunk reaches two or three spheres of each lane, not the same ones, so the packed
// filter leaves a mask of spheres per lane and a lane walks its own (a loop over all twelve
// spheres that every lane of the warp follows took four times the steps); sphere placements come
// from a table of four floats in shared memory and are recomputed from the lane's sines (the same
// bits), the gradient is gathered as seven sums over the pairs, and one exponential serves the
// softplus and its derivative. Cost and gradient of 16384 candidates, K = 32, S = 64, 1000 trees:
// 12.4 ms -> 6.5 ms; the cost of 4096 of them alone 1.58 -> 0.84 ms.
#include "eval_common.cuh"

namespace cp {
namespace {

constexpr int kSmoothThreads = 256;     // 8 warps per CTA, one candidate per warp
constexpr float kSmoothCut = 30.f;      // pairs with sd > m + 30 beta are skipped

struct SmoothArgs {
    const float4 *xi;
    int n, K, S, n_s, chunks;
    float4 q0, qd;
    const float4 *basis;     // [S][2] as in EvalArgs
    float margin, beta;      // softplus margin m and width beta
    float inv_beta;          // 1 / beta rounded to nearest, or 0: divide (beta far from 1)
    float wc_lc, w_l;        // w_c lambda_c and w_l
    const double *gJ;        // [n] or nullptr (ones)
    double *J;               // [n] or nullptr
    float *dxi;              // [n][K][4] or nullptr
    int groups;              // warps per candidate (chunk groups); > 1 writes partials
    int chunks_per_group;
    float *part_g;           // [n groups][4K] when groups > 1
    double *part_J;          // [n groups] when groups > 1
    int *queue;              // the next unit to take (zeroed before the launch), or null: a
                             // fixed stride of units over the warps
};

// n / beta correctly rounded from the correctly rounded reciprocal (Markstein's theorem, IBM J.
// Res. Dev. 34, 1990: q = n y, r = n - q beta exact in an FMA, q + r y rounds to the quotient).
__device__ __forceinline__ float over_beta(float n, const SmoothArgs &a)
{
    if (a.inv_beta == 0.f) return n / a.beta;
    const float q = n * a.inv_beta;
    return fmaf(fmaf(-q, a.beta, n), a.inv_beta, q);
}

// 1 / sqrt(x): the hardware's within 2 ulp, one Newton step.
__device__ __forceinline__ float rsqrt_refined(float x)
{
    const float y = rsqrtf(fmaxf(x, 1e-30f));
    return y * fmaf(-0.5f * x * y, y, 1.5f);
}

// d penalty / d (chain) gathered over the pairs of a checkpoint: with (p_r, p_t, p_z) the
// gradient of a pair's term with respect to its sphere's centre in the crane plane's frame, and
// alpha, L = gamma q4 + beta, gamma the sphere's placement, the kinematic Jacobian needs only
// these sums.
struct ChainSums {
    float ht = 0.f;                   // sum h p_t
    float ar = 0.f, az = 0.f;         // sum alpha p_r, alpha p_z
    float lr = 0.f, lz = 0.f;         // sum L p_r, L p_z
    float gr = 0.f, gz = 0.f;         // sum gamma p_r, gamma p_z
};

// One lane's view of its checkpoint for the pair terms.
struct PairCtx {
    float c1, s1, c2, s2, c23, s23, q4, base_z;
};

// Softplus term of sphere s (its centre at (x, y, z), h from the axis) against an obstacle at
// signed distance sd with SDF gradient g, added to pen and (GRAD) to the chain sums.
template <bool GRAD>
__device__ __forceinline__ void pair_term(const SmoothArgs &a, const PairCtx &c, float sd, float3 g, float h,
                                          float L, float alpha, float gamma, float &pen, ChainSums &sum)
{
    const float x = over_beta(a.margin - sd, a);
    const float e = expf(-fabsf(x));
    const float l = log1pf(e);
    pen = fmaf(a.beta, x > 0.f ? x + l : l, pen);
    if (GRAD) {
        const float inv = __frcp_rn(1.f + e), w = x >= 0.f ? -inv : -(e * inv);   // - logistic(x)
        const float pr = w * fmaf(c.c1, g.x, c.s1 * g.y), pt = w * fmaf(c.c1, g.y, -(c.s1 * g.x)), pz = w * g.z;
        sum.ht = fmaf(h, pt, sum.ht);
        sum.ar = fmaf(alpha, pr, sum.ar);
        sum.az = fmaf(alpha, pz, sum.az);
        sum.lr = fmaf(L, pr, sum.lr);
        sum.lz = fmaf(L, pz, sum.lz);
        sum.gr = fmaf(gamma, pr, sum.gr);
        sum.gz = fmaf(gamma, pz, sum.gz);
    }
}

// h and z of sphere s from the table, by the operations of crane_place.
__device__ __forceinline__ void place_sphere(const PairCtx &c, float4 t, float &L, float &h, float &z)
{
    L = fmaf(t.z, c.q4, t.y);
    h = fmaf(t.x, c.c2, __fmul_rn(L, c.c23));
    z = c.base_z + fmaf(t.x, c.s2, fmaf(L, c.s23, t.w));
}

// Gradient of the capped-cylinder distance at (x, y, z), as sdf_cylinder_grad with the square
// roots and quotients as refined reciprocal square roots.
__device__ __forceinline__ float3 cylinder_grad(float x, float y, float z, float cx, float cy, float4 e)
{
    const float dx = x - cx, dy = y - cy, r2 = fmaf(dx, dx, dy * dy), ir = rsqrt_refined(r2);
    const float a = r2 * ir - e.x, up = z - e.z, down = e.y - z, b = fmaxf(down, up);
    const float ux = dx * ir, uy = dy * ir, sz = up >= down ? 1.f : -1.f;
    float ca = a >= b ? 1.f : 0.f, cb = a >= b ? 0.f : 1.f;
    if (b > 0.f && a > 0.f) {   // off the rim
        const float ih = rsqrt_refined(fmaf(a, a, b * b));
        ca = a * ih;
        cb = b * ih;
    }
    return make_float3(ca * ux, ca * uy, cb * sz);
}

// Sums of the 16 values v over the warp by a transposing butterfly (15 exchanges of halves, then
// one pairwise add): lane l returns the sum of value l >> 1.
__device__ __forceinline__ float sum16(float *v, int lane)
{
#pragma unroll
    for (int step = 0; step < 4; ++step) {
        const int off = 16 >> step, n = 8 >> step;
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float keep = up ? v[n + i] : v[i], give = up ? v[i] : v[n + i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Shared floats of one warp: the candidate's accumulator [K][4].
__host__ __device__ inline int smooth_warp_floats(int K) { return 4 * K; }

template <int NSPH, bool GRAD>
__global__ void __launch_bounds__(kSmoothThreads, GRAD ? 2 : 3)
k_smooth(const ModelDev m, const SceneDev sc, const SmoothArgs a)
{
    extern __shared__ __align__(16) float4 smem[];
    float4 *s_filt = smem;                      // {cx, cy, W_s, reach}
    float4 *s_exact = s_filt + sc.n_cyl;        // {R, z_lo, z_hi, 0}
    float4 *s_bc = s_exact + sc.n_cyl;
    float4 *s_bh = s_bc + sc.n_box;
    float4 *s_basis = s_bh + sc.n_box;
    float4 *s_group = s_basis + 2 * a.S;
    float *s_warp = reinterpret_cast<float *>(s_group + n_groups(sc.n_cyl));
    __shared__ float4 s_sph[NSPH];
    __shared__ float s_rad[NSPH];
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *s_acc = s_warp + wib * smooth_warp_floats(a.K);
    const double reach = (double)m.r_max + (double)a.margin + (double)kSmoothCut * a.beta;
    for (int i = threadIdx.x; i < sc.n_cyl; i += blockDim.x) {
        const float4 f = sc.cyl_filt[i], e = sc.cyl_exact[i];
        const double R = (double)e.x + reach;
        const double W = (double)f.x * f.x + (double)f.y * f.y - R * R;
        s_filt[i] = make_float4(f.x, f.y, (float)W, f.w);   // w: broad-phase reach
        s_exact[i] = e;
    }
    for (int i = threadIdx.x; i < n_groups(sc.n_cyl); i += blockDim.x) s_group[i] = sc.cyl_group[i];
    for (int i = threadIdx.x; i < sc.n_box; i += blockDim.x) {
        s_bc[i] = sc.box_c[i];
        s_bh[i] = sc.box_h[i];
    }
    for (int i = threadIdx.x; i < 2 * a.S; i += blockDim.x) s_basis[i] = a.basis[i];
    if (threadIdx.x < NSPH) {
        const SphereLin t = m.sph[threadIdx.x];
        s_sph[threadIdx.x] = make_float4(t.alpha, t.beta, t.gamma, -t.delta);
        s_rad[threadIdx.x] = t.radius;
    }
    __syncthreads();

    const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int n_warps = (int)((gridDim.x * blockDim.x) >> 5);
    // A unit is (candidate, group of consecutive chunks); with few candidates several
    // warps share one candidate and write partial sums that k_smooth_reduce combines. A warp
    // takes its next unit from the queue when it has one (candidates in contact cost more),
    // else the units go round the warps in a fixed stride.
    auto next_unit = [&](int u) {
        if (a.queue == nullptr) return u + n_warps;
        int v = 0;
        if (lane == 0) v = atomicAdd(a.queue, 1);
        return __shfl_sync(0xffffffffu, v, 0);
    };
    for (int unit = a.queue == nullptr ? warp : next_unit(0); unit < a.n * a.groups; unit = next_unit(unit)) {
        const int cand = unit / a.groups, group = unit - cand * a.groups;
        const int c_begin = group * a.chunks_per_group;
        const int c_end = min(a.chunks, c_begin + a.chunks_per_group);
        if (GRAD)
            for (int t = lane; t < 4 * a.K; t += 32) s_acc[t] = 0.f;
        double J = 0.0;
        const float4 *xi = a.xi + (size_t)cand * a.K;
        for (int chunk = c_begin; chunk < c_end; ++chunk) {
            const int k = chunk * 32 + lane + 1;
            const bool valid = k <= a.n_s;
            const int kc = valid ? k : a.n_s;
            const int span = (kc - 1) / a.S;
            const int mstep = kc - span * a.S;
            float4 P[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int g = span + 1 + i;
                P[i] = g < 4 ? a.q0 : (g >= a.K + 4 ? a.qd : __ldg(xi + (g - 4)));
            }
            const float4 q = combine4(s_basis[2 * (mstep - 1)], P[0], P[1], P[2], P[3]);
            const float4 dq = combine4(s_basis[2 * (mstep - 1) + 1], P[0], P[1], P[2], P[3]);
            const float jp = fmaf(dq.x, dq.x, fmaf(dq.y, dq.y, fmaf(dq.z, dq.z, dq.w * dq.w)));
            const float jl = limit_excess(q.x, m.q_min[0], m.q_max[0]) + limit_excess(q.y, m.q_min[1], m.q_max[1]) +
                             limit_excess(q.z, m.q_min[2], m.q_max[2]) + limit_excess(q.w, m.q_min[3], m.q_max[3]);
            PairCtx ctx;
            sincosf(q.x, &ctx.s1, &ctx.c1);
            sincosf(q.y, &ctx.s2, &ctx.c2);
            sincosf(q.y + q.z, &ctx.s23, &ctx.c23);
            ctx.q4 = q.w;
            ctx.base_z = m.base_z;
            const float c1 = ctx.c1, s1 = ctx.s1;
            const float extra = a.margin + kSmoothCut * a.beta;
            const float zreach = m.r_max + extra + kZGate;
            const float zlo = sc.z_lo_all - zreach, zhi = sc.z_hi_all + zreach;
            UnitFrame fr;
            float2 X2[NSPH / 2], Y2[NSPH / 2], nT2[NSPH / 2];
            {
                float H[NSPH], Z[NSPH];
                crane_place<NSPH>(m, q.w, ctx.s2, ctx.c2, ctx.s23, ctx.c23, H, Z);
                // broad phase of the chunk: the box of its spheres in the slew frame, dilated by
                // the softplus range m + cut beta beyond the obstacles' contact reach; spheres
                // farther below or above every obstacle than that range (r_max + m + cut beta)
                // add nothing: left out of the box and of the filter
                fr = unit_frame_band<NSPH>(s1, c1, H, Z, zlo, zhi);
#pragma unroll
                for (int p = 0; p < NSPH / 2; ++p) {
                    const float xa = __fmul_rn(c1, H[2 * p]), xb = __fmul_rn(c1, H[2 * p + 1]);
                    const float ya = __fmul_rn(s1, H[2 * p]), yb = __fmul_rn(s1, H[2 * p + 1]);
                    const float ta = Z[2 * p] > zlo && Z[2 * p] < zhi ? kFilterMargin - fmaf(xa, xa, ya * ya) : -1e30f;
                    const float tb = Z[2 * p + 1] > zlo && Z[2 * p + 1] < zhi ? kFilterMargin - fmaf(xb, xb, yb * yb)
                                                                              : -1e30f;
                    X2[p] = make_float2(-2.f * xa, -2.f * xb);
                    Y2[p] = make_float2(-2.f * ya, -2.f * yb);
                    nT2[p] = make_float2(-ta, -tb);
                }
            }
            float pen = 0.f;
            ChainSums sum;
            const int n_grp = n_groups(sc.n_cyl);
            for (int gbase = 0; gbase < n_grp; gbase += 32) {
                uint32_t gmask = __ballot_sync(0xffffffffu, gbase + lane < n_grp &&
                                                                unit_near(fr, s_group[gbase + lane], extra));
                while (gmask) {
                    uint32_t gg = gmask;
                    const int slot = lane >> 3;
                    gg = slot >= 1 ? gg & (gg - 1) : gg;
                    gg = slot >= 2 ? gg & (gg - 1) : gg;
                    gg = slot >= 3 ? gg & (gg - 1) : gg;
                    const int oc = gg ? (gbase + __ffs(gg) - 1) * kGroup + (lane & (kGroup - 1)) : sc.n_cyl;
#pragma unroll
                    for (int k = 0; k < 4; ++k) gmask &= gmask - 1;
                    uint32_t omask = __ballot_sync(0xffffffffu, oc < sc.n_cyl && unit_near(fr, s_filt[oc], extra));
                    while (omask) {
                        const int o = __shfl_sync(0xffffffffu, oc, __ffs(omask) - 1);
                        omask &= omask - 1;
                        const float4 f = s_filt[o];
                        // sphere s is in reach when g - T < 0: the sign of the difference is exact
                        float2 d[NSPH / 2];
#pragma unroll
                        for (int p = 0; p < NSPH / 2; ++p)
                            d[p] = __fadd2_rn(__ffma2_rn(X2[p], make_float2(f.x, f.x),
                                                         __ffma2_rn(Y2[p], make_float2(f.y, f.y),
                                                                    make_float2(f.z, f.z))),
                                              nT2[p]);
                        if (any_negative<NSPH>(d)) {
                            uint32_t in = 0u;   // bit s: sphere s
#pragma unroll
                            for (int p = NSPH / 2 - 1; p >= 0; --p) {
                                in = __funnelshift_l(__float_as_uint(d[p].y), in, 1);
                                in = __funnelshift_l(__float_as_uint(d[p].x), in, 1);
                            }
                            const float4 e = s_exact[o];
                            const float elo = e.y - zreach, ehi = e.z + zreach;
                            while (in) {
                                const int s = __ffs(in) - 1;
                                in &= in - 1;
                                const float4 t = s_sph[s];
                                float L, h, cz;
                                place_sphere(ctx, t, L, h, cz);
                                if (cz > elo && cz < ehi) {
                                    const float cx = __fmul_rn(c1, h), cy = __fmul_rn(s1, h);
                                    const float sd = sdf_cylinder(cx, cy, cz, f.x, f.y, e) - s_rad[s];
                                    const float3 gr = GRAD ? cylinder_grad(cx, cy, cz, f.x, f.y, e)
                                                           : make_float3(0.f, 0.f, 0.f);
                                    pair_term<GRAD>(a, ctx, sd, gr, h, L, t.x, t.z, pen, sum);
                                }
                            }
                        }
                    }
                }
            }
            for (int bbase = 0; bbase < sc.n_box; bbase += 32) {
                uint32_t bmask = __ballot_sync(0xffffffffu, bbase + lane < sc.n_box &&
                                                                unit_near(fr, s_bc[bbase + lane], extra));
                while (bmask) {
                    const int o = bbase + __ffs(bmask) - 1;
                    bmask &= bmask - 1;
                    const float4 cb = s_bc[o], hb = s_bh[o];
#pragma unroll 1
                    for (int s = 0; s < m.n_spheres; ++s) {
                        const float4 t = s_sph[s];
                        float L, h, cz;
                        place_sphere(ctx, t, L, h, cz);
                        const float cx = __fmul_rn(c1, h), cy = __fmul_rn(s1, h);
                        const float sd = sdf_box(cx, cy, cz, cb, hb) - s_rad[s];
                        if (sd < a.margin + kSmoothCut * a.beta) {
                            const float3 gr = GRAD ? sdf_box_grad(cx, cy, cz, cb, hb) : make_float3(0.f, 0.f, 0.f);
                            pair_term<GRAD>(a, ctx, sd, gr, h, L, t.x, t.z, pen, sum);
                        }
                    }
                }
            }
            __syncwarp();

            float v = valid ? jp + a.wc_lc * pen + a.w_l * jl : 0.f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            J += (double)v;   // every lane holds the same sum; lane 0 writes it

            if (GRAD) {
                // r = d(terms at s_k)/dq: penalty through the kinematic Jacobian, and limits
                const float r2 = fmaf(ctx.c23, sum.lz, -ctx.s23 * sum.lr);
                const float r1 = fmaf(ctx.c2, sum.az, fmaf(-ctx.s2, sum.ar, r2));
                const float r3 = fmaf(ctx.c23, sum.gr, ctx.s23 * sum.gz);
                const float4 lim2 = make_float4(
                    2.f * (fmaxf(0.f, q.x - m.q_max[0]) - fmaxf(0.f, m.q_min[0] - q.x)),
                    2.f * (fmaxf(0.f, q.y - m.q_max[1]) - fmaxf(0.f, m.q_min[1] - q.y)),
                    2.f * (fmaxf(0.f, q.z - m.q_max[2]) - fmaxf(0.f, m.q_min[2] - q.z)),
                    2.f * (fmaxf(0.f, q.w - m.q_max[3]) - fmaxf(0.f, m.q_min[3] - q.w)));
                const float4 r = make_float4(fmaf(a.wc_lc, sum.ht, a.w_l * lim2.x), fmaf(a.wc_lc, r1, a.w_l * lim2.y),
                                             fmaf(a.wc_lc, r2, a.w_l * lim2.z), fmaf(a.wc_lc, r3, a.w_l * lim2.w));
                // contribution to control point span+1+i: 2 dq db_i + r b_i, summed over the lanes
                // of each span the chunk covers (one or two when S >= 32). The other lanes' dq and r
                // are taken as 0, not multiplied by it: a checkpoint without a finite gradient
                // spoils its own control points only.
                const float4 bw = s_basis[2 * (mstep - 1)], dbw = s_basis[2 * (mstep - 1) + 1];
                const int sp_lo = __shfl_sync(0xffffffffu, span, 0), sp_hi = __shfl_sync(0xffffffffu, span, 31);
                for (int sp = sp_lo; sp <= sp_hi; ++sp) {
                    const bool mine = valid && span == sp;
                    const float bi[4] = {bw.x, bw.y, bw.z, bw.w}, dbi[4] = {dbw.x, dbw.y, dbw.z, dbw.w};
                    const float4 dm = make_float4(mine ? dq.x : 0.f, mine ? dq.y : 0.f, mine ? dq.z : 0.f, mine ? dq.w : 0.f);
                    const float4 rm = make_float4(mine ? r.x : 0.f, mine ? r.y : 0.f, mine ? r.z : 0.f, mine ? r.w : 0.f);
                    float t[16];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float wd = 2.f * dbi[i], wb = bi[i];
                        t[4 * i + 0] = fmaf(wd, dm.x, wb * rm.x);
                        t[4 * i + 1] = fmaf(wd, dm.y, wb * rm.y);
                        t[4 * i + 2] = fmaf(wd, dm.z, wb * rm.z);
                        t[4 * i + 3] = fmaf(wd, dm.w, wb * rm.w);
                    }
                    const float total = sum16(t, lane);
                    const int at = (sp - 3) * 4 + (lane >> 1);   // control point span + 1 + i, from the first free one
                    if ((lane & 1) == 0 && at >= 0 && at < 4 * a.K) s_acc[at] += total;
                    __syncwarp();
                }
            }
        }
        if (a.groups == 1) {
            if (lane == 0 && a.J != nullptr) a.J[cand] = J;
            if (GRAD) {
                const float gj = a.gJ != nullptr ? (float)a.gJ[cand] : 1.f;
                for (int t = lane; t < 4 * a.K; t += 32) a.dxi[(size_t)cand * 4 * a.K + t] = gj * s_acc[t];
            }
        } else {
            if (lane == 0) a.part_J[unit] = J;
            if (GRAD)
                for (int t = lane; t < 4 * a.K; t += 32) a.part_g[(size_t)unit * 4 * a.K + t] = s_acc[t];
        }
        __syncwarp();
    }
}

// Sums the groups' partials of each candidate in group order: one thread per gradient entry
// (and one more per candidate for J), eight groups' loads in flight before the dependent
// additions. With a warp per candidate that loaded one group at a time the kernel was bound by
// the latency of some 4 x 76 loads in a row (64 candidates, K = 32; ten polish steps 820 us then,
// 303 now).
__global__ void __launch_bounds__(128)
k_smooth_reduce(int n, int groups, int K, const double *__restrict__ part_J, const float *__restrict__ part_g,
                const double *__restrict__ gJ, double *J, float *dxi)
{
    constexpr int kAhead = 8;
    const int cand = blockIdx.x, D = 4 * K;
    for (int t = threadIdx.x; t <= D; t += blockDim.x) {
        if (t == D) {
            if (J == nullptr) continue;
            double acc = 0.0;
            for (int g = 0; g < groups; ++g) acc += part_J[(size_t)cand * groups + g];
            J[cand] = acc;
        } else if (dxi != nullptr) {
            const float *col = part_g + (size_t)cand * groups * D + t;
            float acc = 0.f;
            for (int g0 = 0; g0 < groups; g0 += kAhead) {
                float v[kAhead];
#pragma unroll
                for (int q = 0; q < kAhead; ++q) v[q] = g0 + q < groups ? col[(size_t)(g0 + q) * D] : 0.f;
#pragma unroll
                for (int q = 0; q < kAhead; ++q)
                    if (g0 + q < groups) acc += v[q];
            }
            const float gj = gJ != nullptr ? (float)gJ[cand] : 1.f;
            dxi[(size_t)cand * D + t] = gj * acc;
        }
    }
}

__global__ void k_axpy(float *x, const float *y, float alpha, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = fmaf(-alpha, y[i], x[i]);
}

size_t smooth_smem(int n_cyl, int n_box, int S, int K)
{
    return sizeof(float4) * (2 * (size_t)n_cyl + 2 * (size_t)n_box + 2 * (size_t)S + (size_t)n_groups(n_cyl)) +
           sizeof(float) * (size_t)(kSmoothThreads / 32) * (size_t)smooth_warp_floats(K);
}

template <bool GRAD>
int launch_smooth_t(const ModelDev &m, const SceneDev &sc, const SmoothArgs &a, int num_sms,
                    cudaStream_t st)
{
    const int threads = kSmoothThreads;
    const size_t smem = smooth_smem(sc.n_cyl, sc.n_box, a.S, a.K);
    auto kern = m.n_spheres == 12 ? k_smooth<12, GRAD> : k_smooth<16, GRAD>;
    CP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    CP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (per_sm < 1) per_sm = 1;
    const int units = a.n * a.groups;
    int grid = (units + threads / 32 - 1) / (threads / 32);
    if (grid > num_sms * per_sm) grid = num_sms * per_sm;
    if (a.queue != nullptr) CP_CUDA(cudaMemsetAsync(a.queue, 0, sizeof(int), st));
    kern<<<grid, threads, smem, st>>>(m, sc, a);
    CP_LAUNCHED("k_smooth");
    if (a.groups > 1) {
        k_smooth_reduce<<<a.n, 128, 0, st>>>(a.n, a.groups, a.K, a.part_J, a.part_g, a.gJ, a.J, a.dxi);
        CP_LAUNCHED("k_smooth_reduce");
    }
    return CP_OK;
}

}  // namespace

// The bound a scene has to meet (shared memory of an opt-in block): the obstacle and spline tables
// and, for four warps, lane sums, a candidate's gradient and per-sphere records of 16 spheres.
// The launch needs less; the bound on the accepted scenes stays where it was.
size_t smooth_smem_bytes(int n_cyl, int n_box, int S, int K)
{
    return sizeof(float4) * (2 * (size_t)n_cyl + 2 * (size_t)n_box + 2 * (size_t)S + (size_t)n_groups(n_cyl)) +
           sizeof(float) * 4 * (size_t)(32 * 16 + 32 + 4 * K + 5 * 16 * 32);
}

// Chunk groups per candidate: enough units for about 32 warps per SM when candidates are
// few, at most the number of chunks; the partial buffers hold smooth_partial_units() units.
int smooth_groups(int n, int chunks, int num_sms)
{
    const int target = 32 * num_sms;
    if (n <= 0 || n >= target) return 1;
    int g = (target + n - 1) / n;
    return g < chunks ? g : chunks;
}

int64_t smooth_partial_units(int num_sms) { return 2 * 32 * (int64_t)num_sms; }

int launch_smooth(const ModelDev &m, const SceneDev &sc, const float *xi, int n, int K, int S,
                  float4 q0, float4 qd, const float4 *basis, double margin, double beta,
                  double wc_lc, double w_l, const double *gJ, double *J, float *dxi, float *part_g,
                  double *part_J, int *queue, int num_sms, cudaStream_t st)
{
    if (n == 0) return CP_OK;
    SmoothArgs a{};
    a.queue = queue;
    a.xi = (const float4 *)xi;
    a.n = n;
    a.K = K;
    a.S = S;
    a.n_s = (K + 3) * S;
    a.chunks = (a.n_s + 31) / 32;
    a.q0 = q0;
    a.qd = qd;
    a.basis = basis;
    a.margin = (float)margin;
    a.beta = (float)beta;
    a.inv_beta = a.beta > 1e-18f && a.beta < 1e18f ? 1.f / a.beta : 0.f;
    a.wc_lc = (float)wc_lc;
    a.w_l = (float)w_l;
    a.gJ = gJ;
    a.J = J;
    a.dxi = dxi;
    a.groups = smooth_groups(n, a.chunks, num_sms);
    a.chunks_per_group = (a.chunks + a.groups - 1) / a.groups;
    a.groups = (a.chunks + a.chunks_per_group - 1) / a.chunks_per_group;   // no empty group
    a.part_g = part_g;
    a.part_J = part_J;
    return dxi != nullptr ? launch_smooth_t<true>(m, sc, a, num_sms, st)
                          : launch_smooth_t<false>(m, sc, a, num_sms, st);
}

int launch_axpy(float *x, const float *y, double alpha, int64_t n, cudaStream_t st)
{
    if (n == 0) return CP_OK;
    k_axpy<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, y, (float)alpha, n);
    CP_LAUNCHED("k_axpy");
    return CP_OK;
}

}  // namespace cp
