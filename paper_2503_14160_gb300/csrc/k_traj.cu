// Trajectory tracking optimisation (arXiv 2503.14160, Sec. 4.2, Eq. discrete): the planned
// path q*(s) becomes a near-time-optimal trajectory by trapezoidal direct collocation,
//
//     min  t_F + w_s sum_k u_k^T R u_k + w_t sum_k |q_a,k - q*_a,k|^2
//     s.t. x_{k+1} - x_k = h/2 (f_k + f_{k+1}),  x_0 = x_S,  x_N = x_T,  x_min <= x <= x_max,
//
// h = t_F / N, with f the crane dynamics of Sec. 2.1 with the actuated joints' accelerations as
// inputs. The paper's model parameters are not given; the model here has its structure: the
// four actuated joints driven through their accelerations, and two passive swing angles of the
// grapple, a point mass on a rigid link under the tip, whose accelerations follow from the
// Euler-Lagrange equations of a pendulum with an accelerated pivot.
//
// Method (the paper uses IPOPT; the library solves the same problem by): an augmented
// Lagrangian for the equality constraints (defects and end states) and a quadratic penalty
// for the bounds, so that the objective is F(z) = t_F + 1/2 |r(z)|^2 + const; damped
// Gauss-Newton (Levenberg-Marquardt) steps (J^T J + mu (diag J^T J + 1e-9)) dz = -(e_t + J^T r),
// accepted when F decreases (mu / 3, else mu * 4), `inner` of them per multiplier update
// lambda <- lambda + rho c. J^T J is block tridiagonal in the grid points' 16 variables
// w_k = (x_k, u_k) with a border for t_F (the defects couple neighbours and t_F); it is
// factored block by block (16 x 16 Cholesky factors L_k, L_k^-1 E_k) and the border is taken
// through its Schur complement. The dynamics' Jacobian per grid point comes from forward-mode
// differentiation (one derivative per pass, 16 passes). Everything is FP64: a
// cluster of two, four or eight CTAs of 512 threads per trajectory.
//
// What bounds it: the FP64 units. A warp instruction holds its scheduler's unit for 64 cycles
// whatever lanes are active, and a dependent one waits as long, so the work is laid out to issue
// few of them and to spread them over all schedulers of the cluster. Rows 0-9 of df/dw are
// constant (the rates and the inputs), so only rows 10 and 11 are stored and every sum over the 12
// rows takes the terms that are not zero; a warp of the Jacobian takes one variable, so that the
// terms that do not depend on it are left out; quotients are formed once; the block factor
// carries the right-hand sides as further rows on the lanes that a 16-row factor leaves idle;
// warps are numbered across the CTAs; the back substitution reads its blocks from shared memory,
// staged before the barrier. 64 trajectories of 100 intervals (two CTAs each): 164.2 ms with none of
// this, 105.0 ms with the first two and the factor, 75.6 ms with all of it, with the same bits. Of
// an LM step's 1.15 M cycles then the levels' factors take 55%, their updates 30%, the Jacobian 6%.
#include <cmath>
#include <new>
#include <type_traits>

#include <cooperative_groups.h>
#include <nvtx3/nvToolsExt.h>

#include "cp_internal.cuh"
#include "fp64_chain.cuh"

// An NVTX range over a scope (no-op without a profiling tool).
struct NvtxScope {
    explicit NvtxScope(const char *name) { nvtxRangePushA(name); }
    ~NvtxScope() { nvtxRangePop(); }
};

namespace cp {
namespace {

constexpr int kTrajThreads = 512;
constexpr int kSumCtas = 2;       // CTAs of a cluster that take the team sums (see Team)
constexpr int kRedDoubles = 64;   // block reductions: [0, 32) and [32, 64) (one slot per warp)
constexpr int NX = 12, NU = 4, NW = 16;
constexpr int NF = 2;             // dense rows of df/dw (rows NX - NF .. NX - 1)
constexpr int kWarpScratch = 3 * NW * NW + 2 * NW;   // doubles of shared memory per warp (three
                                                     // blocks, two of them with padded rows)
constexpr double kGravity = 9.81;

// A value and one derivative (forward mode).
struct Dual {
    double v, d;
};
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return {a.v + b.v, a.d + b.d}; }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return {a.v - b.v, a.d - b.d}; }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) { return {a.v * b.v, a.d * b.v + a.v * b.d}; }
__device__ __forceinline__ Dual operator*(double s, Dual a) { return {s * a.v, s * a.d}; }
__device__ __forceinline__ Dual operator/(Dual a, Dual b)
{
    const double q = a.v / b.v;
    return {q, (a.d - q * b.d) / b.v};
}
template <typename T> __device__ __forceinline__ T lift(double v);
template <> __device__ __forceinline__ double lift<double>(double v) { return v; }
template <> __device__ __forceinline__ Dual lift<Dual>(double v) { return {v, 0.0}; }

// The same where the seed is known when this is compiled: an operand that does not depend on it is
// a plain double, and its products and quotients leave out the terms that a zero derivative would
// make. What is left is rounded as the full pairs are, each operation by name, so that no fusion
// is left to the compiler: fma(0, x, y) is y and fma(x, y, 0) the rounded product.
struct Part {
    double v, d;
};
__device__ __forceinline__ Part operator+(Part a, Part b) { return {a.v + b.v, __dadd_rn(a.d, b.d)}; }
__device__ __forceinline__ Part operator+(Part a, double b) { return {a.v + b, a.d}; }
__device__ __forceinline__ Part operator+(double a, Part b) { return {a + b.v, b.d}; }
__device__ __forceinline__ Part operator-(Part a, Part b) { return {a.v - b.v, __dadd_rn(a.d, -b.d)}; }
__device__ __forceinline__ Part operator-(Part a, double b) { return {a.v - b, a.d}; }
__device__ __forceinline__ Part operator-(double a, Part b) { return {a - b.v, -b.d}; }
__device__ __forceinline__ Part operator*(Part a, Part b) { return {a.v * b.v, fma(a.v, b.d, __dmul_rn(a.d, b.v))}; }
__device__ __forceinline__ Part operator*(double a, Part b) { return {a * b.v, __dmul_rn(a, b.d)}; }
__device__ __forceinline__ Part operator*(Part a, double b) { return {a.v * b, __dmul_rn(a.d, b)}; }
__device__ __forceinline__ Part operator/(Part a, double b) { return {a.v / b, a.d / b}; }
__device__ __forceinline__ double value(double a) { return a; }
__device__ __forceinline__ double value(Part a) { return a.v; }

// x with the value v
__device__ __forceinline__ double with_value(double, double v) { return v; }
__device__ __forceinline__ Part with_value(Part x, double v) { return {v, x.d}; }

// z + x y and z - x y with the values fused
template <typename X, typename Y, typename Z>
__device__ __forceinline__ auto madd(X x, Y y, Z z)
{
    return with_value(z + x * y, fma(value(x), value(y), value(z)));
}
template <typename X, typename Y, typename Z>
__device__ __forceinline__ auto msub(X x, Y y, Z z)
{
    return with_value(z - x * y, fma(-value(x), value(y), value(z)));
}

// s x + y for a constant s, fused
__device__ __forceinline__ double axpy(double s, double x, double y) { return fma(s, x, y); }
__device__ __forceinline__ Part axpy(double s, Part x, double y) { return {fma(s, x.v, y), __dmul_rn(s, x.d)}; }
__device__ __forceinline__ Part axpy(double s, double x, Part y) { return {fma(s, x, y.v), y.d}; }
__device__ __forceinline__ Part axpy(double s, Part x, Part y) { return {fma(s, x.v, y.v), fma(s, x.d, y.d)}; }

// Variable I of the grid point's 16 (states, then inputs).
template <int SEED, int I>
__device__ __forceinline__ auto seeded(const double *w)
{
    if constexpr (SEED == I) return Part{w[I], 1.0};
    else return w[I];
}

// Cosine and sine of an angle of the dynamics. The primal values depend on the grid point
// only, so a cache (c, s pairs written by the value pass at that point) serves the 16
// derivative passes; without one (or for plain doubles) they are computed here.
__device__ __forceinline__ void trig_of(double a, const double *cache, double *cw, int idx, double &c, double &s)
{
    if (cache != nullptr) {
        c = cache[2 * idx];
        s = cache[2 * idx + 1];
        return;
    }
    sincos(a, &s, &c);
    if (cw != nullptr) {
        cw[2 * idx] = c;
        cw[2 * idx + 1] = s;
    }
}

__device__ __forceinline__ void trig_of(Dual a, const double *cache, double *cw, int idx, Dual &c, Dual &s)
{
    double cv, sv;
    if (cache != nullptr) {
        cv = cache[2 * idx];
        sv = cache[2 * idx + 1];
    } else {
        sincos(a.v, &sv, &cv);
    }
    (void)cw;
    c = {cv, -sv * a.d};
    s = {sv, cv * a.d};
}

__device__ __forceinline__ void trig_of(Part a, const double *cache, double *, int idx, Part &c, Part &s)
{
    const double cv = cache[2 * idx], sv = cache[2 * idx + 1];
    c = {cv, __dmul_rn(-sv, a.d)};
    s = {sv, __dmul_rn(cv, a.d)};
}

struct TrajDev {
    double base_z, boom_len, jib_len, ell;
    double omega_s, omega_t, R[4];
    double x_min[NX], x_max[NX];
    double rho, rho_b, mu0;
    int N, outer, inner;
    double inv_N, inv_2N;   // reciprocals rounded to nearest
};

// a / b correctly rounded from b's correctly rounded reciprocal (Markstein's theorem, IBM J. Res.
// Dev. 34, 1990), three FP64 instructions where a division takes some thirty.
__device__ __forceinline__ double quotient(double a, double b, double inv_b)
{
    const double q = a * inv_b;
    return fma(fma(-q, b, a), inv_b, q);
}

// x' = f(x, u): the actuated joints' rates and accelerations, and the swing accelerations from
// the tip acceleration T'' (cylindrical coordinates of the tip) by
//   (ddalpha, ddbeta) = -(r_a . v / l, r_b . v / (l cos^2 alpha)),  v = T'' + l w + g z,
//   r = (sin a, cos a sin b, -cos a cos b),  w = r_aa da^2 + 2 r_ab da db + r_bb db^2.
// cache: the cosines and sines of this grid point (A, B, q1, alpha, beta) when known; cw: where
// the value pass stores them (either may be null).
template <typename T>
__device__ void traj_f(const TrajDev &td, const T *x, const T *u, T *out, const double *cache = nullptr,
                       double *cw = nullptr)
{
    const T q1 = x[0], q2 = x[1], q3 = x[2], q4 = x[3], a = x[4], b = x[5];
    const T d1 = x[6], d2 = x[7], d3 = x[8], d4 = x[9], da = x[10], db = x[11];
    const T u1 = u[0], u2 = u[1], u3 = u[2], u4 = u[3];
    const T lam = lift<T>(td.jib_len) + q4;
    const T A = q2, B = q2 + q3, dB = d2 + d3, ddB = u2 + u3;
    T cA, sA, cB, sB;
    trig_of(A, cache, cw, 0, cA, sA);
    trig_of(B, cache, cw, 1, cB, sB);
    const T h = td.boom_len * cA + lam * cB;
    const T dh = lift<T>(0.0) - td.boom_len * sA * d2 + d4 * cB - lam * sB * dB;
    const T ddh = lift<T>(0.0) - td.boom_len * (cA * d2 * d2 + sA * u2) + u4 * cB - 2.0 * d4 * sB * dB -
                  lam * (cB * dB * dB + sB * ddB);
    const T ddz = td.boom_len * (cA * u2 - sA * d2 * d2) + u4 * sB + 2.0 * d4 * cB * dB +
                  lam * (cB * ddB - sB * dB * dB);
    const T a_r = ddh - h * d1 * d1, a_t = h * u1 + 2.0 * dh * d1;
    T c1, s1;
    trig_of(q1, cache, cw, 2, c1, s1);
    const T ax = a_r * c1 - a_t * s1, ay = a_r * s1 + a_t * c1;
    T ca, sa, cb, sb;
    trig_of(a, cache, cw, 3, ca, sa);
    trig_of(b, cache, cw, 4, cb, sb);
    // w = r_aa da^2 + 2 r_ab da db + r_bb db^2
    const T wx = lift<T>(0.0) - sa * da * da;
    const T wy = lift<T>(0.0) - ca * sb * da * da - 2.0 * sa * cb * da * db - ca * sb * db * db;
    const T wz = ca * cb * da * da - 2.0 * sa * sb * da * db + ca * cb * db * db;
    const T vx = ax + td.ell * wx, vy = ay + td.ell * wy, vz = ddz + td.ell * wz + lift<T>(kGravity);
    const T ra_v = ca * vx - sa * sb * vy + sa * cb * vz;
    const T rb_v = ca * cb * vy + ca * sb * vz;
    out[0] = d1; out[1] = d2; out[2] = d3; out[3] = d4; out[4] = da; out[5] = db;
    out[6] = u1; out[7] = u2; out[8] = u3; out[9] = u4;
    out[10] = lift<T>(0.0) - ra_v / lift<T>(td.ell);
    out[11] = lift<T>(0.0) - rb_v / (td.ell * ca * ca);
}

// The derivatives of outputs 10 and 11 of traj_f with respect to variable SEED, with the bits of
// traj_f<Dual>: the same expressions over the operands that depend on the seed, the products that a
// sum takes in fused as there (the solver's path follows every bit). Not for the slew angle and the
// swing angles (0, 4, 5), whose derivatives take the accelerations' values.
template <int SEED>
__device__ __noinline__ void swing_deriv(const TrajDev &td, const double *w, const double *cache, double *F10,
                                         double *F11)
{
    static_assert(SEED != 0 && SEED != 4 && SEED != 5);
    double *const cw = nullptr;
    const auto q1 = seeded<SEED, 0>(w);
    const auto q2 = seeded<SEED, 1>(w);
    const auto q3 = seeded<SEED, 2>(w);
    const auto q4 = seeded<SEED, 3>(w);
    const auto a = seeded<SEED, 4>(w);
    const auto b = seeded<SEED, 5>(w);
    const auto d1 = seeded<SEED, 6>(w);
    const auto d2 = seeded<SEED, 7>(w);
    const auto d3 = seeded<SEED, 8>(w);
    const auto d4 = seeded<SEED, 9>(w);
    const auto da = seeded<SEED, 10>(w);
    const auto db = seeded<SEED, 11>(w);
    const auto u1 = seeded<SEED, 12>(w);
    const auto u2 = seeded<SEED, 13>(w);
    const auto u3 = seeded<SEED, 14>(w);
    const auto u4 = seeded<SEED, 15>(w);
    const auto lam = td.jib_len + q4;
    const auto A = q2;
    const auto B = q2 + q3;
    const auto dB = d2 + d3;
    const auto ddB = u2 + u3;
    std::decay_t<decltype(A)> cA, sA;
    std::decay_t<decltype(B)> cB, sB;
    trig_of(A, cache, cw, 0, cA, sA);
    trig_of(B, cache, cw, 1, cB, sB);
    const auto h = with_value(axpy(td.boom_len, cA, lam * cB),
                              fma(value(lam), value(cB), __dmul_rn(td.boom_len, value(cA))));
    const auto dh = msub(lam * sB, dB, madd(d4, cB, 0.0 - td.boom_len * sA * d2));
    const auto bend = madd(sB, ddB, cB * dB * dB);
    const auto rise = madd(cB, ddB, 0.0 - sB * dB * dB);
    const auto ddh = 0.0 - td.boom_len * (cA * d2 * d2 + sA * u2) + u4 * cB - 2.0 * d4 * sB * dB - lam * bend;
    const auto ddz = axpy(td.boom_len, cA * u2 - sA * d2 * d2, u4 * sB) + 2.0 * d4 * cB * dB + lam * rise;
    const auto a_r = ddh - h * d1 * d1;
    const auto a_t = h * u1 + 2.0 * dh * d1;
    std::decay_t<decltype(q1)> c1, s1;
    trig_of(q1, cache, cw, 2, c1, s1);
    const auto ax = a_r * c1 - a_t * s1;
    const auto ay = a_r * s1 + a_t * c1;
    std::decay_t<decltype(a)> ca, sa;
    std::decay_t<decltype(b)> cb, sb;
    trig_of(a, cache, cw, 3, ca, sa);
    trig_of(b, cache, cw, 4, cb, sb);
    // w = r_aa da^2 + 2 r_ab da db + r_bb db^2
    const auto wx = 0.0 - sa * da * da;
    const auto wy = 0.0 - ca * sb * da * da - 2.0 * sa * cb * da * db - ca * sb * db * db;
    const auto wz = ca * cb * da * da - 2.0 * sa * sb * da * db + ca * cb * db * db;
    const auto vx = axpy(td.ell, wx, ax);
    const auto vy = axpy(td.ell, wy, ay);
    const auto vz = axpy(td.ell, wz, ddz) + kGravity;
    const auto ra_v = ca * vx - sa * sb * vy + sa * cb * vz;
    const auto rb_v = ca * cb * vy + ca * sb * vz;
    const auto o10 = 0.0 - ra_v / td.ell;
    const auto o11 = 0.0 - rb_v / (td.ell * ca * ca);
    *F10 = o10.d;
    *F11 = o11.d;
}

__device__ __noinline__ void swing_deriv_any(const TrajDev &td, const double *w, int seed, const double *cache,
                                             double *F10, double *F11)
{
    Dual x[NX], u[NU], out[NX];
#pragma unroll
    for (int i = 0; i < NX; ++i) x[i] = {w[i], i == seed ? 1.0 : 0.0};
#pragma unroll
    for (int i = 0; i < NU; ++i) u[i] = {w[NX + i], NX + i == seed ? 1.0 : 0.0};
    traj_f<Dual>(td, x, u, out, cache);
    *F10 = out[10].d;
    *F11 = out[11].d;
}

// Column `seed` (uniform over the warp) of the dense rows of df/dw at one grid point.
__device__ __forceinline__ void swing_column(const TrajDev &td, const double *w, const double *trig, int seed,
                                             double *F10, double *F11)
{
    switch (seed) {
    case 1: swing_deriv<1>(td, w, trig, F10, F11); break;
    case 2: swing_deriv<2>(td, w, trig, F10, F11); break;
    case 3: swing_deriv<3>(td, w, trig, F10, F11); break;
    case 6: swing_deriv<6>(td, w, trig, F10, F11); break;
    case 7: swing_deriv<7>(td, w, trig, F10, F11); break;
    case 8: swing_deriv<8>(td, w, trig, F10, F11); break;
    case 9: swing_deriv<9>(td, w, trig, F10, F11); break;
    case 10: swing_deriv<10>(td, w, trig, F10, F11); break;
    case 11: swing_deriv<11>(td, w, trig, F10, F11); break;
    case 12: swing_deriv<12>(td, w, trig, F10, F11); break;
    case 13: swing_deriv<13>(td, w, trig, F10, F11); break;
    case 14: swing_deriv<14>(td, w, trig, F10, F11); break;
    case 15: swing_deriv<15>(td, w, trig, F10, F11); break;
    default: swing_deriv_any(td, w, seed, trig, F10, F11); break;
    }
}

// Per-trajectory device workspace (doubles), laid out by the launcher.
struct TrajWs {
    double *f;     // [N+1][12]
    double *Fj;    // [N+1][2][16] rows 10 and 11 of df/dw (row r < 10: 1 at column r + 6)
    double *D;     // [N+1][16][16] diagonal blocks, then their Cholesky factors
    double *E;     // [N][16][16] off-diagonal blocks, then L_k^-1 E_k
    double *bb;    // [N+1][16] border column, then the forward/back solves
    double *g;     // [N+1][16] gradient, then the forward/back solves
    double *P;     // [N+1][16][16] L_k^-1 T[k][left neighbour] of the eliminated blocks
    double *trig;  // [N+1][10] cosines and sines of the dynamics at the grid points of z
    double *er;    // [N][12] d(defect)/dt_F
    double *dr;    // [N][12] defect + lambda / rho
    double *b0;    // [N+1][16] border column as assembled
    double *lr;    // [N+2][12] lambda / rho
};

__device__ __forceinline__ TrajWs ws_of(double *base, int N)
{
    TrajWs w;
    w.f = base;
    w.Fj = w.f + (size_t)(N + 1) * NX;
    w.D = w.Fj + (size_t)(N + 1) * NF * NW;
    w.E = w.D + (size_t)(N + 1) * NW * NW;
    w.bb = w.E + (size_t)N * NW * NW;
    w.g = w.bb + (size_t)(N + 1) * NW;
    w.P = w.g + (size_t)(N + 1) * NW;
    w.trig = w.P + (size_t)(N + 1) * NW * NW;
    w.er = w.trig + (size_t)(N + 1) * 10;
    w.dr = w.er + (size_t)N * NX;
    w.b0 = w.dr + (size_t)N * NX;
    w.lr = w.b0 + (size_t)(N + 1) * NW;
    return w;
}

// The CTAs of one trajectory: a cluster of 2, 4 or 8 CTAs on neighbouring SMs. Grid points,
// entries and blocks are split over the team-wide thread or warp index. Data one CTA writes to
// the trajectory's global workspace is read by the other only after team_sync(), a cluster
// barrier with release / acquire semantics. Every thread of both CTAs passes the same
// sequence of them: no barrier sits under a branch whose condition the CTAs could see
// differently (the sums below give all the same values). Sums over the trajectory are taken by
// the first kSumCtas CTAs alone, whatever the cluster's size, so that their order, and with it
// every bit of the solution, does not depend on how many trajectories share the GPU; they are
// under 2% of the work.
struct Team {
    int rank;   // this CTA's rank in the cluster
    int ctas;   // CTAs in the cluster
    // warps are numbered across the CTAs, so that a level of few blocks has them on all SMs
    __device__ int warp() const { return ((int)threadIdx.x >> 5) * ctas + rank; }
    __device__ int nwarps() const { return ctas * (int)blockDim.x >> 5; }
    __device__ int tid() const { return warp() * 32 + ((int)threadIdx.x & 31); }
    __device__ int nthreads() const { return ctas * (int)blockDim.x; }
    // this thread's first term and the stride of a team sum (no term on the other CTAs)
    __device__ int sum_first(int n) const { return rank < kSumCtas ? rank * (int)blockDim.x + (int)threadIdx.x : n; }
    __device__ int sum_stride() const { return kSumCtas * (int)blockDim.x; }
};

__device__ __forceinline__ Team team_of_block()
{
    const cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    return Team{(int)cl.block_rank(), (int)cl.num_blocks()};
}

__device__ __forceinline__ void team_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Sums of a and b over the two summing CTAs in a fixed order: per warp by shuffles, a CTA's
// warps in order by its thread 0, then CTA 0's partial plus CTA 1's (read from each CTA's shared
// memory), so every thread of the cluster returns the same values (deterministic).
__device__ double2 team_sum2(double a, double b, double *s_red)
{
    const int t = threadIdx.x;
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
    }
    __syncthreads();
    if ((t & 31) == 0) {
        s_red[t >> 5] = a;
        s_red[32 + (t >> 5)] = b;
    }
    __syncthreads();
    if (t == 0) {
        double sa = 0.0, sb = 0.0;
        for (int i = 0; i < kTrajThreads / 32; ++i) {
            sa += s_red[i];
            sb += s_red[32 + i];
        }
        s_red[kRedDoubles - 2] = sa;
        s_red[kRedDoubles - 1] = sb;
    }
    team_sync();   // both CTAs' partials are written
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const double *p0 = cl.map_shared_rank(s_red + kRedDoubles - 2, 0);
    const double *p1 = cl.map_shared_rank(s_red + kRedDoubles - 2, 1);
    const double2 r = make_double2(p0[0] + p1[0], p0[1] + p1[1]);
    team_sync();   // every thread has read them before either CTA writes s_red again
    return r;
}

__device__ double team_sum(double v, double *s_red) { return team_sum2(v, 0.0, s_red).x; }

// f at every grid point of z (values only) into ws.f, the points split over the team.
// trig (optional): the cosines and sines of every grid point are stored there too.
__device__ void eval_f(const Team &tm, const TrajDev &td, const double *z, double *f, double *trig = nullptr)
{
    for (int k = tm.tid(); k <= td.N; k += tm.nthreads()) {
        const double *w = z + 1 + (size_t)k * NW;
        traj_f<double>(td, w, w + NX, f + (size_t)k * NX, nullptr, trig != nullptr ? trig + (size_t)k * 10 : nullptr);
    }
}

// The merit F(z) = t_F + 1/2 |r(z)|^2 (T6): the AL terms of the defects and end states, the
// effort and tracking sums over k = 1..N, and the bound penalty; f must be current for z.
__device__ double merit(const Team &tm, const TrajDev &td, const double *z, const double *lam_rho, const double *q_star,
                        const double *f, const double *x_S, const double *x_T, double *s_red)
{
    const int N = td.N;
    const double h = quotient(z[0], N, td.inv_N);
    double acc = 0.0;
    // defects and end states: rho/2 (c + lam/rho)^2
    for (int e = tm.sum_first(NX * (N + 2)); e < NX * (N + 2); e += tm.sum_stride()) {
        const int k = e / NX, i = e - k * NX;
        double c;
        if (k < N) {
            const double *w0 = z + 1 + (size_t)k * NW, *w1 = w0 + NW;
            c = w1[i] - w0[i] - 0.5 * h * (f[(size_t)k * NX + i] + f[(size_t)(k + 1) * NX + i]);
        } else if (k == N) {
            c = z[1 + i] - x_S[i];
        } else {
            c = z[1 + (size_t)N * NW + i] - x_T[i];
        }
        const double t = c + lam_rho[e];
        acc += 0.5 * td.rho * t * t;
    }
    // effort, tracking and bounds per grid point
    for (int e = tm.sum_first((N + 1) * NW); e < (N + 1) * NW; e += tm.sum_stride()) {
        const int k = e / NW, i = e - k * NW;
        const double v = z[1 + e];
        if (i < NX) {
            const double lo = td.x_min[i], hi = td.x_max[i];
            const double viol = v > hi ? v - hi : (v < lo ? v - lo : 0.0);
            acc += 0.5 * td.rho_b * viol * viol;
            if (i < 4 && k >= 1) {
                const double dq = v - q_star[(size_t)k * 4 + i];
                acc += td.omega_t * dq * dq;
            }
        } else if (k >= 1) {
            acc += td.omega_s * td.R[i - NX] * v * v;
        }
    }
    return z[0] + team_sum(acc, s_red);
}

// Elimination of one 16 x 16 SPD block A = L L^T on one warp, with its right-hand sides riding
// along: P = L^-1 Tl, Q = L^-1 Tr and y = L^-1 f for the two vectors. A row of a right-hand
// side's transpose takes the same operations as a row of A below the pivot, so the lanes hold
//   lanes 0-15   row i of A, and column i of Tr;
//   lanes 16-31  column c of Tl, and (lanes 16, 17) the two vectors,
// one row in each of two register sets: per pivot one reciprocal square root (rsqrt_newton), one
// scaling and one FMA per later column and set, with the pivot's column from shuffles. That is
// about 400 FP64 warp instructions and one chain of 16 pivots where the factor followed by three
// column solves took 710 and three more chains. Tl is the transpose of Tl_rows (row-major
// 16 x 16); Q overwrites Tr, the vectors are solved in place, and A's block receives the strict
// lower triangle of L with 1 / L_pp on the diagonal. P, Tl_rows or Tr may be null.
__device__ __noinline__ void warp_eliminate16(double *A, const double *Tl_rows, double *P, double *Tr, double *f_y,
                                              double *f_v, int lane)
{
    const unsigned full = 0xffffffffu;
    const int i = lane & (NW - 1);
    const bool low = lane < NW;
    double *f = lane == NW ? f_y : f_v;
    double a[NW], b[NW], diag = 0.0;
#pragma unroll
    for (int j = 0; j < NW; ++j) {
        a[j] = low ? (j <= i ? A[i * NW + j] : 0.0) : (Tl_rows != nullptr ? Tl_rows[i * NW + j] : 0.0);
        b[j] = low ? (Tr != nullptr ? Tr[j * NW + i] : 0.0) : (i < 2 ? f[j] : 0.0);
    }
#pragma unroll
    for (int p = 0; p < NW; ++p) {
        const double d = __shfl_sync(full, a[p], p);   // the pivot, from lane p
        const double r = rsqrt_newton(d);
        double l = a[p] * r;                            // L[i][p], or P[p][i]
        if (low && i <= p) l = i == p ? d * r : 0.0;
        if (lane == p) diag = r;
        a[p] = l;
        const double l2 = b[p] * r;
        b[p] = l2;
#pragma unroll
        for (int j = p + 1; j < NW; ++j) {
            const double lj = __shfl_sync(full, l, j);  // L[j][p]
            a[j] = fma(-l, lj, a[j]);
            b[j] = fma(-l2, lj, b[j]);
        }
    }
    __syncwarp();
    if (low) {
#pragma unroll
        for (int j = 0; j < NW; ++j) A[i * NW + j] = j < i ? a[j] : (j == i ? diag : 0.0);
    } else if (P != nullptr) {
#pragma unroll
        for (int j = 0; j < NW; ++j) P[j * NW + i] = a[j];
    }
    if (low) {
        if (Tr != nullptr) {
#pragma unroll
            for (int j = 0; j < NW; ++j) Tr[j * NW + i] = b[j];
        }
    } else if (i < 2) {
#pragma unroll
        for (int j = 0; j < NW; ++j) f[j] = b[j];
    }
    __syncwarp();
}

// A block of the back substitution in the warp's shared memory: L_k as it is, P_k and Q_k with rows
// of 17 doubles, so that lanes of different rows read different banks. Coalesced loads, all in
// flight together; issued before the barrier that the neighbours' solutions wait for.
constexpr int kPadRow = NW + 1, kPadBlock = NW * kPadRow;

__device__ __forceinline__ void stage_back(double *sm, const double *Lk, const double *P, const double *Q, int lane)
{
    double *sP = sm + NW * NW, *sQ = sP + kPadBlock;
#pragma unroll
    for (int q = 0; q < NW * NW / 32; ++q) {
        const int e = q * 32 + lane, at = (e >> 4) * kPadRow + (e & (NW - 1));
        sm[e] = Lk[e];
        if (P != nullptr) sP[at] = P[e];
        if (Q != nullptr) sQ[at] = Q[e];
    }
    __syncwarp();
}

// x_k = L_k^-T (w_k - P_k x_l - Q_k x_r) for both vectors (lanes 0-15 y, 16-31 v, one row
// each; P or Q absent when has_p or has_q is false), the block staged by stage_back: the products,
// then L^T x = rhs from the last row up, column by column with the solved entry shuffled to the
// rows above it.
__device__ __noinline__ void warp_back16(const double *sm, bool has_p, const double *xl_y, const double *xl_v,
                                         bool has_q, const double *xr_y, const double *xr_v, double *out_y,
                                         double *out_v, int lane)
{
    const unsigned full = 0xffffffffu;
    const int r = lane & (NW - 1), which = lane >> 4, first = NW * which;
    const double *sP = sm + NW * NW, *sQ = sP + kPadBlock;
    double *out = which ? out_v : out_y;
    const double xl = has_p ? (which ? xl_v : xl_y)[r] : 0.0, xq = has_q ? (which ? xr_v : xr_y)[r] : 0.0;
    double x = out[r];   // w_k
    if (has_p) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int c = 0; c < NW; c += 2) {
            s0 = fma(sP[r * kPadRow + c], __shfl_sync(full, xl, first + c), s0);
            s1 = fma(sP[r * kPadRow + c + 1], __shfl_sync(full, xl, first + c + 1), s1);
        }
        x -= s0 + s1;
    }
    if (has_q) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int c = 0; c < NW; c += 2) {
            s0 = fma(sQ[r * kPadRow + c], __shfl_sync(full, xq, first + c), s0);
            s1 = fma(sQ[r * kPadRow + c + 1], __shfl_sync(full, xq, first + c + 1), s1);
        }
        x -= s0 + s1;
    }
#pragma unroll
    for (int rr = NW - 1; rr >= 0; --rr) {
        const double lrr = sm[rr * NW + rr];     // 1 / L_rr
        const double lrq = sm[rr * NW + r];      // L[rr][r] (r < rr)
        const double xr = __shfl_sync(full, x * lrr, rr + first);
        if (r == rr) x = xr;
        else if (r < rr) x = fma(-lrq, xr, x);
    }
    __syncwarp();
    out[r] = x;
    __syncwarp();
}

// The damped Gauss-Newton step dz at z (T6): Jacobian, assembly, block factorisation, solve.
// dz_local: dz is this CTA's shared-memory copy, which gets every entry; otherwise it is one
// global vector whose entries the team splits.
__device__ void lm_step(const Team &tm, const TrajDev &td, const double *z, const double *q_star,
                        const double *x_S, const double *x_T, double mu, const TrajWs &ws, double *dz, bool dz_local,
                        double *s_red, double *s_blk)
{
    const int N = td.N, t = tm.tid(), nt = tm.nthreads();
    const double h = quotient(z[0], N, td.inv_N), rho = td.rho;
    // 1. f and df/dw at every grid point
    eval_f(tm, td, z, ws.f, ws.trig);
    team_sync();
    // a warp takes one seed at 32 grid points; the dear seeds (slew and swing angles, angles and
    // rates of the arm) come first and the cheap ones in the reverse order, so that a warp that
    // takes two has one of each
    {
        const unsigned long long order = 0xFCED6BA938721540ull;   // seed of place i: bits 4 i ..
        const int groups = (N + 32) / 32, lane = threadIdx.x & 31;
        for (int m = tm.warp(); m < NW * groups; m += tm.nwarps()) {
            const int seed = (int)(order >> (4 * (m / groups))) & 15, k = 32 * (m % groups) + lane;
            if (k <= N) {
                double *F = ws.Fj + (size_t)k * NF * NW + seed;
                swing_column(td, z + 1 + (size_t)k * NW, ws.trig + (size_t)k * 10, seed, F, F + NW);
            }
        }
    }
    // defect k: e_k = dd_k/dt_F = -(f_k + f_{k+1}) / (2N) and d_k + lam_k / rho
    for (int e = t; e < N * NX; e += nt) {
        const int k = e / NX, r = e - k * NX;
        const double *w0 = z + 1 + (size_t)k * NW;
        const double fs = ws.f[e] + ws.f[e + NX];
        ws.er[e] = quotient(-fs, 2.0 * N, td.inv_2N);
        ws.dr[e] = w0[NW + r] - w0[r] - 0.5 * h * fs + ws.lr[e];
    }
    team_sync();
    // 2. assembly. Defect k: d_k = x_{k+1} - x_k - h/2 (f_k + f_{k+1}), rows scaled by sqrt(rho):
    //    A_k = dd_k/dw_k = -[I 0] - h/2 Fj_k, B_k = dd_k/dw_{k+1} = [I 0] - h/2 Fj_{k+1},
    //    e_k = dd_k/dt_F = -(f_k + f_{k+1}) / (2N); residual sqrt(rho) (d_k + lam_k / rho).
    // Diagonal blocks (lower triangles) and off-diagonal blocks from F_k = df/dw at grid
    // point k (c = h/2, I' = [I 0] of 12 x 16): A_k = -(I' + c F_k), B_k = I' - c F_{k+1}, so
    //   A_k^T A_k = I'^T I' + c (I'^T F_k + F_k^T I') + c^2 F_k^T F_k,
    //   B_{k-1}^T B_{k-1} = I'^T I' - c (I'^T F_k + F_k^T I') + c^2 F_k^T F_k
    // (interior points take both, whose first-order terms cancel) and
    //   A_k^T B_k = -(I'^T I' - c I'^T F_{k+1} + c F_k^T I' - c^2 F_k^T F_{k+1}).
    const double c = 0.5 * h, cc = c * c;
    // one warp per grid point k: rows 10 and 11 of F_k and F_{k+1} staged in the warp's shared
    // memory, then the 136 lower entries of D_k and the 256 of E_k. Row r < 10 of F adds 1 to a
    // product's entry (r + 6, r + 6) and nothing elsewhere.
    {
        const int warp = tm.warp(), lane = threadIdx.x & 31, n_warps = tm.nwarps();
        double *sF = s_blk + (size_t)(threadIdx.x >> 5) * kWarpScratch;   // [2][NF][NW]: F_k, F_{k+1}
        const double *F0 = sF, *F1 = sF + NF * NW;
        auto Fent = [&](const double *F, int r, int i) -> double {
            return r < NX - NF ? (i == r + 6 ? 1.0 : 0.0) : F[(r - (NX - NF)) * NW + i];
        };
        for (int k = warp; k <= N; k += n_warps) {
            __syncwarp();
            for (int q = lane; q < 2 * NF * NW; q += 32)
                sF[q] = (q < NF * NW || k < N) ? ws.Fj[(size_t)k * NF * NW + q] : 0.0;
            __syncwarp();
            const bool end = k == 0 || k == N;
            const double ck = k == 0 ? c : -c, s = end ? cc : 2.0 * cc;
            for (int e = lane; e < NW * (NW + 1) / 2; e += 32) {
                int i, j;
                tri_index(e, i, j);
                const bool one = i == j && i >= 6;
                const double ff = fma(F0[i], F0[j], one && (i & 1) == 0 ? 1.0 : 0.0) +             // even rows
                                  fma(F0[NW + i], F0[NW + j], one && (i & 1) != 0 ? 1.0 : 0.0);    // odd rows
                double v = i == j && i < NX ? (end ? 1.0 : 2.0) : 0.0;
                if (end) v = fma(ck, (i < NX ? Fent(F0, i, j) : 0.0) + (j < NX ? Fent(F0, j, i) : 0.0), v);
                ws.D[(size_t)k * NW * NW + i * NW + j] = fma(s, ff, v) * rho;
            }
            __syncwarp();
            if (lane < NW) {   // what only the diagonal has
                const int i = lane;
                double *d = &ws.D[(size_t)k * NW * NW + i * (NW + 1)], v = *d;
                if (end && i < NX) v += rho;                                          // end states
                if (i < NX) {
                    const double x = z[1 + (size_t)k * NW + i];
                    if (x > td.x_max[i] || x < td.x_min[i]) v += td.rho_b;        // active bound
                    if (i < 4 && k >= 1) v += 2.0 * td.omega_t;                   // tracking
                } else if (k >= 1) {
                    v += 2.0 * td.omega_s * td.R[i - NX];                         // effort
                }
                *d = v + mu * (v + 1e-9);                                         // damping
            }
            if (k < N)
#pragma unroll
                for (int q = 0; q < NW * NW / 32; ++q) {
                    const int e = q * 32 + lane, i = e >> 4, j = e & (NW - 1);
                    const bool one = i == j && i >= 6, dense = q == (NX - NF) / 2;   // rows 10 and 11
                    const double p = fma(F0[i], F1[j], one && (i & 1) == 0 ? 1.0 : 0.0) +
                                     fma(F0[NW + i], F1[NW + j], one && (i & 1) != 0 ? 1.0 : 0.0);
                    // I'^T I' - c I'^T F_(k+1) + c F_k^T I': ones of the constant rows by selection
                    const bool below = i == j + 6 && j < NX - NF;
                    double v = i == j && i < NX ? 1.0 : (j == i + 6 && i < NX - NF ? -c : (below ? c : 0.0));
                    if (dense) {
                        v = fma(-c, F1[(lane >> 4) * NW + j], i == j ? 1.0 : 0.0);
                        if (below) v += c;
                    }
                    if (j == NX - 2 || j == NX - 1) v = fma(c, F0[(j - (NX - NF)) * NW + i], v);
                    v = -rho * fma(-cc, p, v);
                    ws.E[(size_t)k * NW * NW + e] = v;
                }
        }
    }
    // border column, gradient (stored negated: the solves below take -g): column i of A_k^T and
    // B_{k-1}^T has entries in rows i - 6 (the constant rows of F), i and the two dense rows
    for (int e = t; e < (N + 1) * NW; e += nt) {
        const int k = e / NW, i = e - k * NW;
        double bv = 0.0, gv = 0.0;
        auto add = [&](double a, size_t at) {
            bv = fma(a, ws.er[at], bv);
            gv = fma(a, ws.dr[at], gv);
        };
        const double *Fk = ws.Fj + (size_t)k * NF * NW;
        if (k < N) {   // A_k = -[I 0] - h/2 F_k
            const size_t at = (size_t)k * NX;
            if (i >= 6) add(-0.5 * h, at + i - 6);
            if (i < NX - NF) add(-1.0, at + i);
            add((i == NX - 2 ? -1.0 : 0.0) - 0.5 * h * Fk[i], at + NX - 2);
            add((i == NX - 1 ? -1.0 : 0.0) - 0.5 * h * Fk[NW + i], at + NX - 1);
        }
        if (k > 0) {   // B_{k-1} = [I 0] - h/2 F_k
            const size_t at = (size_t)(k - 1) * NX;
            if (i >= 6) add(-0.5 * h, at + i - 6);
            if (i < NX - NF) add(1.0, at + i);
            add((i == NX - 2 ? 1.0 : 0.0) - 0.5 * h * Fk[i], at + NX - 2);
            add((i == NX - 1 ? 1.0 : 0.0) - 0.5 * h * Fk[NW + i], at + NX - 1);
        }
        bv *= rho;
        gv *= rho;
        const double x = z[1 + e];
        if (i < NX) {
            if (k == 0) gv += rho * (x - x_S[i] + ws.lr[(size_t)N * NX + i]);
            if (k == N) gv += rho * (x - x_T[i] + ws.lr[(size_t)(N + 1) * NX + i]);
            const double viol = x > td.x_max[i] ? x - td.x_max[i] : (x < td.x_min[i] ? x - td.x_min[i] : 0.0);
            gv += td.rho_b * viol;
            if (i < 4 && k >= 1) gv += 2.0 * td.omega_t * (x - q_star[(size_t)k * 4 + i]);
        } else if (k >= 1) {
            gv += 2.0 * td.omega_s * td.R[i - NX] * x;
        }
        ws.bb[e] = bv;
        ws.b0[e] = bv;
        ws.g[e] = -gv;
    }
    // the t_F corner and gradient
    double ct = 0.0, gt = 0.0;
    for (int e = tm.sum_first(N * NX); e < N * NX; e += tm.sum_stride()) {
        const double ev = ws.er[e];
        ct += ev * ev;
        gt += ev * ws.dr[e];
    }
    {
        const double2 sums = team_sum2(ct, gt, s_red);   // also orders D, E, bb, g before the solve
        ct = rho * sums.x;
        gt = 1.0 + rho * sums.y;
    }
    ct += mu * (ct + 1e-9);
    // 3. the tridiagonal part T (diagonal blocks D_k, couplings T[k][k+1] = E_k) solved for the
    //    two right-hand sides b (into y, ws.bb) and -g (into v, ws.g) by block cyclic reduction.
    //    Level s = 1, 2, 4, ... eliminates the blocks k = s, 3s, 5s, ... <= N, each between
    //    l = k - s and r = k + s (when r <= N), one warp per block:
    //      L L^T = D_k,  P = L^-1 T[k][l],  Q = L^-1 T[k][r],  w = L^-1 f_k,
    //    then the kept blocks j = 0, 2s, 4s, ... take D_j -= Q_(j-s)^T Q_(j-s) + P_(j+s)^T P_(j+s),
    //    f_j -= Q_(j-s)^T w_(j-s) + P_(j+s)^T w_(j+s) and the coupling T'[j][j+2s] = -P^T Q of
    //    block j + s. Block 0 is left and solved; the eliminated blocks then follow level by
    //    level from the last: x_k = L^-T (w - P x_l - Q x_r). The couplings are kept in ws.E
    //    under their left block (E_l becomes the new coupling; E_k then holds Q), P in ws.P,
    //    the factors (1 / L_pp on the diagonal) in ws.D, w and x in ws.bb / ws.g. Each level's
    //    blocks are independent, so the chain of dependent FP64 steps is that of about
    //    log2(N + 1) block factors instead of N + 1.
    const int warp = tm.warp(), lane = threadIdx.x & 31, n_warps = tm.nwarps();
    double *Fw = s_blk + (size_t)(threadIdx.x >> 5) * kWarpScratch;
    int s_top = 1;
    for (int s = 1; s <= N; s <<= 1) {
        s_top = s;
        const int n_odd = (N / s + 1) / 2;
        for (int m = warp; m < n_odd; m += n_warps) {   // phase A
            const int k = (2 * m + 1) * s, l = k - s, r = k + s;
            const bool has_r = r <= N;
            // T[k][l] is the transpose of the coupling E_l; T[k][r] = E_k becomes Q in place
            warp_eliminate16(ws.D + (size_t)k * NW * NW, ws.E + (size_t)l * NW * NW, ws.P + (size_t)k * NW * NW,
                             has_r ? ws.E + (size_t)k * NW * NW : nullptr, ws.bb + (size_t)k * NW,
                             ws.g + (size_t)k * NW, lane);
        }
        team_sync();
        const int n_even = N / (2 * s) + 1;
        for (int m = warp; m < n_even; m += n_warps) {   // phase B
            const int j = 2 * m * s, iL = j - s, iR = j + s;
            const bool hasL = m > 0, hasR = iR <= N;
            const bool hasE = hasR && iR + s <= N;
            // Q_(j-s), P_(j+s) and Q_(j+s) staged in the warp's shared memory (coalesced loads,
            // all in flight together), the 136 lower entries packed over the lanes
            double *QL = Fw, *PR = Fw + NW * NW, *QR = Fw + 2 * NW * NW;
            const double2 *gQL = reinterpret_cast<const double2 *>(ws.E + (size_t)(hasL ? iL : 0) * NW * NW);
            const double2 *gPR = reinterpret_cast<const double2 *>(ws.P + (size_t)(hasR ? iR : 0) * NW * NW);
            const double2 *gQR = reinterpret_cast<const double2 *>(ws.E + (size_t)(hasE ? iR : 0) * NW * NW);
#pragma unroll
            for (int q = 0; q < NW * NW / 64; ++q) {
                const int at = q * 32 + lane;
                if (hasL) reinterpret_cast<double2 *>(QL)[at] = gQL[at];
                if (hasR) reinterpret_cast<double2 *>(PR)[at] = gPR[at];
                if (hasE) reinterpret_cast<double2 *>(QR)[at] = gQR[at];
            }
            __syncwarp();
            for (int e = lane; e < NW * (NW + 1) / 2; e += 32) {
                int a, b;
                tri_index(e, a, b);
                double *d = ws.D + (size_t)j * NW * NW + a * NW + b;
                double v0 = *d, v1 = 0.0;
                if (hasL)
#pragma unroll
                    for (int q = 0; q < NW; ++q) v0 = fma(-QL[q * NW + a], QL[q * NW + b], v0);
                if (hasR)
#pragma unroll
                    for (int q = 0; q < NW; ++q) v1 = fma(-PR[q * NW + a], PR[q * NW + b], v1);
                *d = v0 + v1;
            }
            {
                const int a = lane & (NW - 1), which = lane >> 4;
                double *f = which ? ws.g : ws.bb;
                double v = f[(size_t)j * NW + a];
                if (hasL) {
                    const double *w = f + (size_t)iL * NW;
#pragma unroll
                    for (int q = 0; q < NW; ++q) v = fma(-QL[q * NW + a], w[q], v);
                }
                if (hasR) {
                    const double *w = f + (size_t)iR * NW;
#pragma unroll
                    for (int q = 0; q < NW; ++q) v = fma(-PR[q * NW + a], w[q], v);
                }
                f[(size_t)j * NW + a] = v;
            }
            if (hasE) {
                for (int e = lane; e < NW * NW; e += 32) {
                    const int a = e >> 4, b = e & (NW - 1);
                    double v = 0.0;
#pragma unroll
                    for (int q = 0; q < NW; ++q) v = fma(PR[q * NW + a], QR[q * NW + b], v);
                    ws.E[(size_t)j * NW * NW + e] = -v;
                }
            }
            __syncwarp();
        }
        team_sync();
    }
    // block 0: D_0 x_0 = f_0; then the eliminated blocks, from the last level to the first. Each
    // warp stages its first block of the next level before the barrier.
    auto stage_level = [&](int s, int m) {
        const int n_odd = (N / s + 1) / 2;
        if (m >= n_odd) return;
        const int k = (2 * m + 1) * s;
        stage_back(Fw, ws.D + (size_t)k * NW * NW, ws.P + (size_t)k * NW * NW,
                   k + s <= N ? ws.E + (size_t)k * NW * NW : nullptr, lane);
    };
    if (warp == 0) {
        warp_eliminate16(ws.D, nullptr, nullptr, nullptr, ws.bb, ws.g, lane);
        stage_back(Fw, ws.D, nullptr, nullptr, lane);
        warp_back16(Fw, false, nullptr, nullptr, false, nullptr, nullptr, ws.bb, ws.g, lane);
    }
    stage_level(s_top, warp);
    team_sync();
    for (int s = s_top; s >= 1; s >>= 1) {
        const int n_odd = (N / s + 1) / 2;
        for (int m = warp; m < n_odd; m += n_warps) {
            const int k = (2 * m + 1) * s, l = k - s, r = k + s;
            const bool has_r = r <= N;
            if (m != warp) stage_level(s, m);
            warp_back16(Fw, true, ws.bb + (size_t)l * NW, ws.g + (size_t)l * NW, has_r,
                        ws.bb + (size_t)(has_r ? r : 0) * NW, ws.g + (size_t)(has_r ? r : 0) * NW,
                        ws.bb + (size_t)k * NW, ws.g + (size_t)k * NW, lane);
        }
        if (s > 1) stage_level(s >> 1, warp);
        team_sync();
    }
    // 4. the border: dt = (-g_t - b^T v) / (c - b^T y), dw = v - y dt, with y = T^-1 b and
    //    v = T^-1 (-g_w), b the border column as assembled.
    double by = 0.0, bv = 0.0;
    for (int e = tm.sum_first((N + 1) * NW); e < (N + 1) * NW; e += tm.sum_stride()) {
        const double b = ws.b0[e];
        by += b * ws.bb[e];
        bv += b * ws.g[e];
    }
    const double2 sums = team_sum2(by, bv, s_red);
    by = sums.x;
    bv = sums.y;
    const double dt = (-gt - bv) / (ct - by);
    const int d0 = dz_local ? (int)threadIdx.x : t, dn = dz_local ? (int)blockDim.x : nt;
    if (d0 == 0) dz[0] = dt;
    for (int e = d0; e < (N + 1) * NW; e += dn) dz[1 + e] = ws.g[e] - ws.bb[e] * dt;
    __syncthreads();
}

// One LM step for each trajectory (a test of the step): dz at (z, lam, mu). Cluster p of
// CTAS CTAs serves trajectory p.
template <int CTAS>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(kTrajThreads)
k_traj_step(const TrajDev td, const double *q_star, const double *z, const double *lam, double mu, double *ws_base,
            size_t ws_stride, double *dz)
{
    extern __shared__ double s_mem[];
    const int N = td.N, n_var = 1 + NW * (N + 1), n_eq = NX * (N + 2);
    const int p = (int)(blockIdx.x / CTAS);
    const Team tm = team_of_block();
    double *s_red = s_mem;                                      // kRedDoubles
    double *s_blk = s_red + kRedDoubles;                        // per warp kWarpScratch
    double *x_S = s_blk + (kTrajThreads / 32) * kWarpScratch, *x_T = x_S + NX;
    const double *qs = q_star + (size_t)p * (N + 1) * 4;
    for (int i = threadIdx.x; i < NX; i += blockDim.x) {
        x_S[i] = i < 4 ? qs[i] : 0.0;
        x_T[i] = i < 4 ? qs[(size_t)N * 4 + i] : 0.0;
    }
    const TrajWs ws = ws_of(ws_base + (size_t)p * ws_stride, N);
    for (int i = tm.tid(); i < n_eq; i += tm.nthreads()) ws.lr[i] = lam[(size_t)p * n_eq + i] / td.rho;
    team_sync();
    lm_step(tm, td, z + (size_t)p * n_var, qs, x_S, x_T, mu, ws, dz + (size_t)p * n_var, false, s_red, s_blk);
}

// The whole solve (T6) for each trajectory: z in place; stats {t_F, F, max |c|, max bound
// violation}. Cluster p of CTAS CTAs serves trajectory p; each CTA keeps z, the trial
// point and the step in its shared memory and updates all of them itself (the same values in
// all), the multipliers and the workspace are global and split.
template <int CTAS>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(kTrajThreads)
k_traj_solve(const TrajDev td, const double *q_star, double *z_io, double *ws_base, size_t ws_stride, double *lam_ws,
             double *stats)
{
    extern __shared__ double s_mem[];
    const int N = td.N, n_var = 1 + NW * (N + 1), n_eq = NX * (N + 2);
    const int p = (int)(blockIdx.x / CTAS), t = threadIdx.x;
    const Team tm = team_of_block();
    double *s_red = s_mem;
    double *s_blk = s_red + kRedDoubles;
    double *x_S = s_blk + (kTrajThreads / 32) * kWarpScratch, *x_T = x_S + NX;
    double *z = x_T + NX;          // n_var
    double *zn = z + n_var;        // n_var
    double *dz = zn + n_var;       // n_var
    double *lam = lam_ws + (size_t)p * n_eq;
    const double *qs = q_star + (size_t)p * (N + 1) * 4;
    for (int i = t; i < NX; i += blockDim.x) {
        x_S[i] = i < 4 ? qs[i] : 0.0;
        x_T[i] = i < 4 ? qs[(size_t)N * 4 + i] : 0.0;
    }
    for (int i = t; i < n_var; i += blockDim.x) z[i] = z_io[(size_t)p * n_var + i];
    const TrajWs ws = ws_of(ws_base + (size_t)p * ws_stride, N);
    for (int i = tm.tid(); i < n_eq; i += tm.nthreads()) {
        lam[i] = 0.0;
        ws.lr[i] = 0.0;
    }
    team_sync();
    double mu = td.mu0;
    for (int o = 0; o < td.outer; ++o) {
        eval_f(tm, td, z, ws.f);
        team_sync();
        double F = merit(tm, td, z, ws.lr, qs, ws.f, x_S, x_T, s_red);
        for (int it = 0; it < td.inner; ++it) {
            lm_step(tm, td, z, qs, x_S, x_T, mu, ws, dz, true, s_red, s_blk);
            for (int i = t; i < n_var; i += blockDim.x) zn[i] = z[i] + dz[i];
            __syncthreads();
            eval_f(tm, td, zn, ws.f);
            team_sync();
            const double Fn = merit(tm, td, zn, ws.lr, qs, ws.f, x_S, x_T, s_red);
            if (Fn < F) {
                for (int i = t; i < n_var; i += blockDim.x) z[i] = zn[i];
                F = Fn;
                mu = fmax(quotient(mu, 3.0, 1.0 / 3.0), 1e-12);
            } else {
                mu = fmin(mu * 4.0, 1e12);
            }
            __syncthreads();
        }
        // multipliers: lam += rho c(z)
        eval_f(tm, td, z, ws.f);
        team_sync();
        const double h = quotient(z[0], N, td.inv_N);
        for (int e = tm.tid(); e < n_eq; e += tm.nthreads()) {
            const int k = e / NX, i = e - k * NX;
            double c;
            if (k < N) c = z[1 + (size_t)(k + 1) * NW + i] - z[1 + (size_t)k * NW + i] -
                           0.5 * h * (ws.f[(size_t)k * NX + i] + ws.f[(size_t)(k + 1) * NX + i]);
            else if (k == N) c = z[1 + i] - x_S[i];
            else c = z[1 + (size_t)N * NW + i] - x_T[i];
            const double l = lam[e] + td.rho * c;
            lam[e] = l;
            ws.lr[e] = l / td.rho;
        }
        team_sync();
    }
    // results and statistics (each CTA takes every entry; CTA 0 writes them)
    if (tm.rank == 0)
        for (int i = t; i < n_var; i += blockDim.x) z_io[(size_t)p * n_var + i] = z[i];
    eval_f(tm, td, z, ws.f);
    team_sync();
    double cmax = 0.0, vmax = 0.0;
    const double h = quotient(z[0], N, td.inv_N);
    for (int e = t; e < n_eq; e += blockDim.x) {
        const int k = e / NX, i = e - k * NX;
        double c;
        if (k < N) c = z[1 + (size_t)(k + 1) * NW + i] - z[1 + (size_t)k * NW + i] -
                       0.5 * h * (ws.f[(size_t)k * NX + i] + ws.f[(size_t)(k + 1) * NX + i]);
        else if (k == N) c = z[1 + i] - x_S[i];
        else c = z[1 + (size_t)N * NW + i] - x_T[i];
        cmax = fmax(cmax, fabs(c));
    }
    for (int e = t; e < (N + 1) * NW; e += blockDim.x) {
        const int i = e % NW;
        if (i < NX) {
            const double x = z[1 + e];
            vmax = fmax(vmax, fmax(x - td.x_max[i], td.x_min[i] - x));
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        cmax = fmax(cmax, __shfl_down_sync(0xffffffffu, cmax, off));
        vmax = fmax(vmax, __shfl_down_sync(0xffffffffu, vmax, off));
    }
    __syncthreads();
    if ((t & 31) == 0) {
        s_red[t >> 5] = cmax;
        s_red[32 + (t >> 5)] = vmax;
    }
    __syncthreads();
    if (t == 0 && tm.rank == 0) {
        double c = 0.0, v = 0.0;
        for (int i = 0; i < kTrajThreads / 32; ++i) {
            c = fmax(c, s_red[i]);
            v = fmax(v, s_red[32 + i]);
        }
        stats[(size_t)p * 4 + 2] = c;
        stats[(size_t)p * 4 + 3] = fmax(v, 0.0);
    }
    __syncthreads();
    const double Fend = merit(tm, td, z, ws.lr, qs, ws.f, x_S, x_T, s_red);
    if (t == 0 && tm.rank == 0) {
        stats[(size_t)p * 4 + 0] = z[0];
        stats[(size_t)p * 4 + 1] = Fend;
    }
}

// q*(k / N) of cubic B-spline paths with control points ctrl[n][K+8][4] on the moving spans
// (tau = 4 + (K+3) s on uniform knots, the path step's reading), by the uniform cubic basis
// of the span that holds tau (s = 1 falls on the last moving span at u = 1).
__global__ void k_traj_targets(const double *ctrl, int K, int n, int N, double *q_star)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * (N + 1)) return;
    const int p = e / (N + 1), k = e - p * (N + 1);
    const double tau = 4.0 + (double)(K + 3) * ((double)k / (double)N);
    int span = (int)floor(tau);
    if (span > K + 6) span = K + 6;        // s = 1: u = 1 on the last moving span
    const double u = tau - span, v = 1.0 - u;
    const double b0 = v * v * v / 6.0, b1 = (3.0 * u * u * u - 6.0 * u * u + 4.0) / 6.0;
    const double b2 = (-3.0 * u * u * u + 3.0 * u * u + 3.0 * u + 1.0) / 6.0, b3 = u * u * u / 6.0;
    const double *P = ctrl + (size_t)p * (K + 8) * 4 + (size_t)(span - 3) * 4;
    for (int j = 0; j < 4; ++j)
        q_star[(size_t)e * 4 + j] = b0 * P[j] + b1 * P[4 + j] + b2 * P[8 + j] + b3 * P[12 + j];
}

// The initial guess of T6 from the targets: q_a = q*_k, dq by central differences over t_F,
// u by second differences, the swing at rest; t_F = 1.5 x the slowest joint's total variation
// over its velocity limit.
__global__ void k_traj_initial(const TrajDev td, const double *dq_max, const double *q_star, int n, double *z)
{
    const int p = blockIdx.x, N = td.N, n_var = 1 + NW * (N + 1);
    if (p >= n) return;
    const double *qs = q_star + (size_t)p * (N + 1) * 4;
    __shared__ double s_tF;
    if (threadIdx.x == 0) {
        double tf = 0.0;
        for (int j = 0; j < 4; ++j) {
            double tv = 0.0;
            for (int k = 0; k < N; ++k) tv += fabs(qs[(size_t)(k + 1) * 4 + j] - qs[(size_t)k * 4 + j]);
            tf = fmax(tf, 1.5 * tv / dq_max[j]);
        }
        s_tF = fmax(tf, 1e-3);
    }
    __syncthreads();
    const double tF = s_tF, h = tF / N;
    double *zp = z + (size_t)p * n_var;
    if (threadIdx.x == 0) zp[0] = tF;
    for (int e = threadIdx.x; e < (N + 1) * NW; e += blockDim.x) {
        const int k = e / NW, i = e - k * NW;
        double v = 0.0;
        if (i < 4) v = qs[(size_t)k * 4 + i];
        else if (i >= 6 && i < 10 && k > 0 && k < N)
            v = (qs[(size_t)(k + 1) * 4 + i - 6] - qs[(size_t)(k - 1) * 4 + i - 6]) / (2.0 * h);
        else if (i >= NX && k > 0 && k < N)
            v = (qs[(size_t)(k + 1) * 4 + i - NX] - 2.0 * qs[(size_t)k * 4 + i - NX] + qs[(size_t)(k - 1) * 4 + i - NX]) /
                (h * h);
        zp[1 + e] = v;
    }
}

}  // namespace
}  // namespace cp

using namespace cp;

struct cp_traj {
    cudaStream_t st = nullptr;
    TrajDev td{};
    int max_paths = 0;
    size_t ws_stride = 0;   // doubles per trajectory
    int fit4 = 0, fit8 = 0; // clusters of 4 and of 8 CTAs the device holds at a time
    double *ws = nullptr, *lam = nullptr, *dq_max = nullptr;
};

namespace {

size_t traj_ws_doubles(int N)
{
    return (size_t)(N + 1) * (NX + NF * NW + 2 * NW * NW + 3 * NW + 10) + (size_t)N * (NW * NW + 2 * NX) +
           (size_t)NX * (N + 2);
}

size_t traj_smem(int N, bool solve);

// Clusters of `ctas` CTAs of the solver that the device holds at a time.
template <int CTAS>
cudaError_t resident_clusters(int N, int *count)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = CTAS;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(CTAS);
    cfg.blockDim = dim3(kTrajThreads);
    cfg.dynamicSmemBytes = traj_smem(N, true);
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(count, k_traj_solve<CTAS>, &cfg);
}

size_t traj_smem(int N, bool solve)
{
    const size_t base = kRedDoubles + (size_t)(kTrajThreads / 32) * kWarpScratch + 2 * NX;
    return sizeof(double) * (base + (solve ? 3 * (size_t)(1 + NW * (N + 1)) : 0));
}

}  // namespace

extern "C" {

int cp_traj_init(const cp_model *model, const cp_traj_params *tp, int32_t max_paths, void *stream, cp_traj **out)
{
    if (!out) return set_error("out is NULL"), CP_ERR_ARG;
    *out = nullptr;
    int rc = validate_model(model);
    if (rc != CP_OK) return rc;
    if (!tp) return set_error("params is NULL"), CP_ERR_ARG;
    if (tp->N < 2 || tp->N > 255) return set_error("N %d outside 2..255", tp->N), CP_ERR_ARG;
    if (max_paths < 1) return set_error("max_paths must be >= 1"), CP_ERR_ARG;
    if (tp->outer < 0 || tp->inner < 0) return set_error("outer and inner must be >= 0"), CP_ERR_ARG;
    if (!(tp->grapple_len > 0.0) || !(tp->rho > 0.0) || !(tp->rho_b >= 0.0) || !(tp->mu0 > 0.0) ||
        !(tp->omega_s >= 0.0) || !(tp->omega_t >= 0.0) || !(tp->swing_max > 0.0) || tp->swing_max >= 1.5)
        return set_error("trajectory weights and limits out of range"), CP_ERR_ARG;
    for (int j = 0; j < 4; ++j)
        if (!(tp->dq_max[j] > 0.0) || !(tp->R[j] >= 0.0)) return set_error("dq_max must be > 0, R >= 0"), CP_ERR_ARG;
    if (traj_smem(tp->N, true) > 227 * 1024) return set_error("N too large for the solver's shared memory"), CP_ERR_ARG;
    cp_traj *t = new (std::nothrow) cp_traj();
    if (!t) return set_error("host allocation failed"), CP_ERR_OOM;
    t->st = (cudaStream_t)stream;
    TrajDev &d = t->td;
    d.base_z = model->base_z;
    d.boom_len = model->boom_len;
    d.jib_len = model->jib_len;
    d.ell = tp->grapple_len;
    d.omega_s = tp->omega_s;
    d.omega_t = tp->omega_t;
    for (int j = 0; j < 4; ++j) d.R[j] = tp->R[j];
    for (int j = 0; j < 4; ++j) {
        d.x_min[j] = model->q_min[j];
        d.x_max[j] = model->q_max[j];
        d.x_min[6 + j] = -tp->dq_max[j];
        d.x_max[6 + j] = tp->dq_max[j];
    }
    d.x_min[4] = d.x_min[5] = -tp->swing_max;
    d.x_max[4] = d.x_max[5] = tp->swing_max;
    d.x_min[10] = d.x_min[11] = -1e30;
    d.x_max[10] = d.x_max[11] = 1e30;
    d.rho = tp->rho;
    d.rho_b = tp->rho_b;
    d.mu0 = tp->mu0;
    d.N = tp->N;
    d.outer = tp->outer;
    d.inner = tp->inner;
    d.inv_N = 1.0 / tp->N;
    d.inv_2N = 1.0 / (2.0 * tp->N);
    t->max_paths = max_paths;
    t->ws_stride = (traj_ws_doubles(tp->N) + 31) & ~(size_t)31;
    const size_t n_eq = (size_t)NX * (tp->N + 2);
    const size_t bytes = sizeof(double) * (t->ws_stride * max_paths + n_eq * max_paths + 4);
    cudaError_t e = cudaMalloc((void **)&t->ws, bytes);
    if (e != cudaSuccess) {
        delete t;
        return cuda_fail(e, "cudaMalloc(trajectory workspace)");
    }
    t->lam = t->ws + t->ws_stride * max_paths;
    t->dq_max = t->lam + n_eq * max_paths;
    e = cudaMemcpyAsync(t->dq_max, tp->dq_max, sizeof(double) * 4, cudaMemcpyHostToDevice, t->st);
    // the limit of the largest N: solvers of several sizes share the kernels
    const int smem = (int)traj_smem(255, true);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_traj_solve<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_traj_solve<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_traj_solve<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_traj_step<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = resident_clusters<4>(tp->N, &t->fit4);
    if (e == cudaSuccess) e = resident_clusters<8>(tp->N, &t->fit8);
    if (e == cudaSuccess) e = cudaStreamSynchronize(t->st);
    if (e != cudaSuccess) {
        cudaFree(t->ws);
        delete t;
        return cuda_fail(e, "trajectory solver set-up");
    }
    *out = t;
    return CP_OK;
}

void cp_traj_destroy(cp_traj *t)
{
    if (!t) return;
    cudaStreamSynchronize(t->st);
    cudaFree(t->ws);
    delete t;
}

int cp_traj_targets(cp_traj *t, const double *d_ctrl, int32_t K, int32_t n, double *d_q_star)
{
    if (!t) return set_error("solver is NULL"), CP_ERR_ARG;
    if (K < 1 || K > CP_MAX_WAYPOINTS || n < 0) return set_error("K or n out of range"), CP_ERR_ARG;
    if (n > 0 && (!d_ctrl || !d_q_star)) return set_error("NULL argument"), CP_ERR_ARG;
    if (n == 0) return CP_OK;
    const int total = n * (t->td.N + 1);
    k_traj_targets<<<(total + 127) / 128, 128, 0, t->st>>>(d_ctrl, K, n, t->td.N, d_q_star);
    CP_LAUNCHED("k_traj_targets");
    return CP_OK;
}

int cp_traj_initial_guess(cp_traj *t, const double *d_q_star, int32_t n, double *d_z)
{
    if (!t) return set_error("solver is NULL"), CP_ERR_ARG;
    if (n < 0 || n > t->max_paths) return set_error("n = %d outside 0..%d", n, t->max_paths), CP_ERR_ARG;
    if (n > 0 && (!d_q_star || !d_z)) return set_error("NULL argument"), CP_ERR_ARG;
    if (n == 0) return CP_OK;
    k_traj_initial<<<n, 128, 0, t->st>>>(t->td, t->dq_max, d_q_star, n, d_z);
    CP_LAUNCHED("k_traj_initial");
    return CP_OK;
}

int cp_traj_step(cp_traj *t, const double *d_q_star, int32_t n, const double *d_z, const double *d_lam, double mu,
                 double *d_dz)
{
    const NvtxScope range("craneplan:traj_step");
    if (!t) return set_error("solver is NULL"), CP_ERR_ARG;
    if (n < 0 || n > t->max_paths) return set_error("n = %d outside 0..%d", n, t->max_paths), CP_ERR_ARG;
    if (n > 0 && (!d_q_star || !d_z || !d_lam || !d_dz)) return set_error("NULL argument"), CP_ERR_ARG;
    if (!(mu >= 0.0)) return set_error("mu must be >= 0"), CP_ERR_ARG;
    if (n == 0) return CP_OK;
    k_traj_step<2><<<n * 2, kTrajThreads, traj_smem(t->td.N, false), t->st>>>(t->td, d_q_star, d_z, d_lam, mu,
                                                                                 t->ws, t->ws_stride, d_dz);
    CP_LAUNCHED("k_traj_step");
    return CP_OK;
}

int cp_traj_solve(cp_traj *t, const double *d_q_star, int32_t n, double *d_z, double *d_stats)
{
    const NvtxScope range("craneplan:traj_solve");
    if (!t) return set_error("solver is NULL"), CP_ERR_ARG;
    if (n < 0 || n > t->max_paths) return set_error("n = %d outside 0..%d", n, t->max_paths), CP_ERR_ARG;
    if (n > 0 && (!d_q_star || !d_z || !d_stats)) return set_error("NULL argument"), CP_ERR_ARG;
    if (n == 0) return CP_OK;
    // CTAs per trajectory: the most of 8, 4 or 2 with which every cluster is resident at once (a
    // second wave would cost more than the split gives). The results do not depend on it.
    const int ctas = n <= t->fit8 ? 8 : (n <= t->fit4 ? 4 : 2);
    auto kern = ctas == 8 ? k_traj_solve<8> : (ctas == 4 ? k_traj_solve<4> : k_traj_solve<2>);
    kern<<<n * ctas, kTrajThreads, traj_smem(t->td.N, true), t->st>>>(t->td, d_q_star, d_z, t->ws, t->ws_stride,
                                                                     t->lam, d_stats);
    CP_LAUNCHED("k_traj_solve");
    return CP_OK;
}

}  // extern "C"
