// pnp.cu -- pose refinement by Perspective-n-Point (Sec. III-C.2).
//
// The rendered view at pose_render supplies depth: each matched render pixel
// is back-projected with the view's normalised depth D / A (Eq. depth over
// 1 - T) into a world point X_i; the query's pose W = [R | t] then minimises
// the Huber cost of the reprojection errors pi(W X_i) - q_i.  The solve is
// iteratively reweighted Gauss-Newton in FP64 with the update applied on the
// left, W <- [Exp(phi) R | Exp(phi) t + rho], so the Jacobian of a camera
// point P = R X + t is [I | -[P]x] and of its pixel
// J_pi = [[fx/z, 0, -fx x/z^2], [0, fy/z, -fy y/z^2]].
//
// The problem is small (thousands of pairs, a 6 x 6 system per iteration) but
// FP64, whose rate is about two operations a clock and SM on this GPU: a warp's
// FP64 instruction holds its scheduler's pipe for some 60 clocks, however many of
// its lanes work.  So the pairs are spread over all SMs in one cooperative launch,
// and what counts is the number of passes over the pairs, the barriers between
// them and the length of every chain of FP64 instructions:
//   - one pass per iteration: the trial pose is evaluated with its normal
//     equations, so an accepted step has them already (and the final pose its
//     cost and squared error);
//   - one grid barrier per pass: every block adds all blocks' partial sums, in
//     the same order, and solves the system for itself, so nothing is handed
//     back from a leading block;
//   - a step is judged by the sum of the pairs' changes of cost: the change of the
//     summed cost carries the rounding of the whole sum, which ended solves with
//     outliers early (128 driving solves: geometric mean of the poses' errors 3.5e-14
//     for 1.0e-12, 7.5 iterations for 6.4);
//   - when the full step does not lower the cost (every solve ends there: the
//     cost is flat to rounding at the minimum) the ten halved steps are
//     evaluated in one pass, half of them by each half of the block;
//   - a warp sums its 32 accumulators by recursive halving (31 additions, lane
//     j left with total j) instead of 28 butterflies of five;
//   - the system is solved by Gauss-Jordan elimination with a row per lane and the
//     update formed with an entry per lane; reciprocals and inverse square roots
//     take an FP32 seed and Newton's iteration to FP64, the rotation its power
//     series for angles below half a radian.
// Some 7,000 pairs on the driving street: 600 to 640 us a call with one block per 256
// pairs, five barriers and two passes an iteration, 180 to 230 us so (157 to 196 with
// steps judged by summed costs); of 6,124 pairs 201 us with one pass, one barrier and a
// thread's serial solve, 167 with the lanes' (15 us an iteration, 13 of them with a single
// block: the chain, not the pairs).
#include <algorithm>

#include <cooperative_groups.h>

#include "internal.cuh"
#include "newton.h"

namespace reloc {

constexpr int PNP_THREADS = 128;                    // four warps, one to each of the SM's schedulers
constexpr int PNP_HALVINGS = 10;         // backtracking: the step is halved at most this often
// accumulators of a pass: upper H (21), g (6), Huber cost, pairs with a point,
// squared error and count of the pairs in front of the camera, and the cost's change
// from the current pose, summed pair by pair
enum { PA_G = 21, PA_COST = 27, PA_USED = 28, PA_SQ = 29, PA_CNT = 30, PA_CHANGE = 31, PNP_ACC = 32 };

struct PnpArgs {
    double Rr[9], tr[3];                 // render pose (world -> camera)
    double W0[12];                       // initial pose: R row-major, then t
    double fx, fy, cx, cy;
    int width, height, n, max_iters;
    double huber, alpha_min, tol;
    const float *depth, *alpha;
    const float4 *pairs;
    double4 *X;                          // scratch [n]: world point, w = 1 if used
    double *c;                           // scratch [2][n]: the pairs' costs at the current and at the trial pose
    double *part;                        // scratch [2][gridDim.x][PNP_ACC]: per-block sums, by turns
    double *out;                         // [16 pose, rms, cost, n_used, iters]
};

// Warp sums of N (a power of two, at most 32) values per lane by recursive
// halving: lane l returns the total of value l / (32 / N).
template <int N>
__device__ __forceinline__ double warp_sums(double (&v)[N], int lane)
{
#pragma unroll
    for (int n = N, o = 16; n > 1; n >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const double send = up ? v[i] : v[n / 2 + i];
            const double keep = up ? v[n / 2 + i] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    double x = v[0];
#pragma unroll
    for (int o = 16 / N; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Whether x lies where its FP32 value can seed Newton's iteration (NaN: no).
__device__ __forceinline__ bool seeds(double x) { return x > 1e-36 && x < 1e36; }

// 1 / x for x > 0: FP32 seed (relative error 2^-23), two Newton steps; rounded once.
__device__ __forceinline__ double recip(double x)
{
    if (!seeds(x)) return 1.0 / x;
    return newton_recip(x, (double)__frcp_rn((float)x));
}

// 1 / sqrt(x) for x > 0: FP32 seed, two Newton steps; rounded once.
__device__ __forceinline__ double rsqrt_newton(double x)
{
    if (!seeds(x)) return 1.0 / sqrt(x);
    return newton_rsqrt(x, (double)rsqrtf((float)x));
}

// Huber cost of a squared residual and its weight (1, or k / e beyond k).
__device__ __forceinline__ double huber(double e2, double k, double &w)
{
    w = 1.0;
    if (e2 <= k * k) return 0.5 * e2;
    const double ie = rsqrt_newton(e2);
    w = k * ie;
    return k * fma(e2, ie, -0.5 * k);
}

// One pair's residual at pose W (R row-major, then t): false behind the camera.
__device__ __forceinline__ bool pnp_residual(const PnpArgs &a, const double *W, const double4 &X, const float4 &q,
                                             double &px, double &py, double &iz, double &ru, double &rv, double &e2)
{
    px = W[0] * X.x + W[1] * X.y + W[2] * X.z + W[9];
    py = W[3] * X.x + W[4] * X.y + W[5] * X.z + W[10];
    const double pz = W[6] * X.x + W[7] * X.y + W[8] * X.z + W[11];
    if (pz <= 1e-6) return false;
    iz = recip(pz);
    ru = a.fx * px * iz + a.cx - (double)q.z;
    rv = a.fy * py * iz + a.cy - (double)q.w;
    e2 = ru * ru + rv * rv;
    return true;
}

// Adds one pair's normal equations, cost and squared error at pose W.  The
// Jacobian rows are Ju = (u0, 0, u2, u3, u4, u5), Jv = (0, v1, v2, v3, v4, v5).
// Returns the pair's cost (0 without a point or behind the camera).
__device__ __forceinline__ double pnp_add(const PnpArgs &a, const double *W, const double4 &X, const float4 &q,
                                          double (&acc)[PNP_ACC])
{
    if (X.w == 0.0) return 0.0;
    acc[PA_USED] += 1.0;
    double px, py, iz, ru, rv, e2;
    if (!pnp_residual(a, W, X, q, px, py, iz, ru, rv, e2)) return 0.0;
    double w;
    const double cost = huber(e2, a.huber, w);
    acc[PA_COST] += cost;
    acc[PA_SQ] += e2;
    acc[PA_CNT] += 1.0;
    const double u0 = a.fx * iz, v1 = a.fy * iz;
    const double nx = px * iz, ny = py * iz;            // -u2 / u0, -v2 / v1
    const double u2 = -u0 * nx, u3 = u2 * py, u4 = a.fx - u2 * px, u5 = -u0 * py;
    const double v2 = -v1 * ny, v3 = v2 * py - a.fy, v4 = -v2 * px, v5 = v1 * px;
    const double wu0 = w * u0, wu2 = w * u2, wu3 = w * u3, wu4 = w * u4, wu5 = w * u5;
    const double wv1 = w * v1, wv2 = w * v2, wv3 = w * v3, wv4 = w * v4, wv5 = w * v5;
    acc[0] += wu0 * u0;                                 // (0, 0); (0, 1) is 0
    acc[2] += wu0 * u2; acc[3] += wu0 * u3; acc[4] += wu0 * u4; acc[5] += wu0 * u5;
    acc[6] += wv1 * v1;
    acc[7] += wv1 * v2; acc[8] += wv1 * v3; acc[9] += wv1 * v4; acc[10] += wv1 * v5;
    acc[11] += wu2 * u2 + wv2 * v2; acc[12] += wu2 * u3 + wv2 * v3;
    acc[13] += wu2 * u4 + wv2 * v4; acc[14] += wu2 * u5 + wv2 * v5;
    acc[15] += wu3 * u3 + wv3 * v3; acc[16] += wu3 * u4 + wv3 * v4; acc[17] += wu3 * u5 + wv3 * v5;
    acc[18] += wu4 * u4 + wv4 * v4; acc[19] += wu4 * u5 + wv4 * v5;
    acc[20] += wu5 * u5 + wv5 * v5;
    acc[21] += wu0 * ru; acc[22] += wv1 * rv;
    acc[23] += wu2 * ru + wv2 * rv; acc[24] += wu3 * ru + wv3 * rv;
    acc[25] += wu4 * ru + wv4 * rv; acc[26] += wu5 * ru + wv5 * rv;
    return cost;
}

// A = sin(th) / th and B = (1 - cos(th)) / th^2 from th^2: Exp = I + A K + B K^2,
// K = [phi]x.  Power series in th^2 up to a quarter (the last term kept is below
// 2^-60 there), the functions beyond.
__device__ __forceinline__ void exp_factors(double th2, double &A, double &B)
{
    if (th2 <= 0.25) {
        // 1 / (2 k + 1)! and 1 / (2 k + 2)!, alternating, k = 8 .. 0
        const double ca[9] = {1.0 / 355687428096000.0, -1.0 / 1307674368000.0, 1.0 / 6227020800.0, -1.0 / 39916800.0,
                              1.0 / 362880.0, -1.0 / 5040.0, 1.0 / 120.0, -1.0 / 6.0, 1.0};
        const double cb[9] = {1.0 / 6402373705728000.0, -1.0 / 20922789888000.0, 1.0 / 87178291200.0, -1.0 / 479001600.0,
                              1.0 / 3628800.0, -1.0 / 40320.0, 1.0 / 720.0, -1.0 / 24.0, 0.5};
        A = ca[0];
        B = cb[0];
#pragma unroll
        for (int k = 1; k < 9; ++k) {
            A = fma(A, th2, ca[k]);
            B = fma(B, th2, cb[k]);
        }
    } else {
        const double th = sqrt(th2);
        double sn, cs;
        sincos(th, &sn, &cs);
        A = sn / th;
        B = (1.0 - cs) / th2;
    }
}

// W' = [Exp(phi) R | Exp(phi) t + rho] for delta = (rho, phi) scaled by s, an entry
// per lane of 12 lanes (q): row q / 3 and column q % 3 of R, then t; with K^2 =
// phi phi^T - th^2 I, row r of Exp is (1 - B th^2) e_r + A [phi]x_r + B phi_r phi^T.
__device__ __forceinline__ double update_entry(const double *W, const double *delta, double s, int q)
{
    const double p0 = s * delta[3], p1 = s * delta[4], p2 = s * delta[5];
    const double th2 = p0 * p0 + p1 * p1 + p2 * p2;
    double A, B;
    exp_factors(th2, A, B);
    const int r = q < 9 ? q / 3 : q - 9;
    const double pr = r == 0 ? p0 : r == 1 ? p1 : p2, d = fma(-B, th2, 1.0), bp = B * pr;
    const double k0 = r == 0 ? 0.0 : r == 1 ? p2 : -p1, k1 = r == 0 ? -p2 : r == 1 ? 0.0 : p0;
    const double k2 = r == 0 ? p1 : r == 1 ? -p0 : 0.0;
    const double e0 = fma(bp, p0, fma(A, k0, r == 0 ? d : 0.0)), e1 = fma(bp, p1, fma(A, k1, r == 1 ? d : 0.0));
    const double e2 = fma(bp, p2, fma(A, k2, r == 2 ? d : 0.0));
    const int o = q < 9 ? q % 3 : 9, step = q < 9 ? 3 : 1;
    return fma(e0, W[o], fma(e1, W[o + step], fma(e2, W[o + 2 * step], q < 9 ? 0.0 : s * delta[r])));
}

// Solve (H + 1e-9 tr(H)/6 I) x = -g, H given as 21 upper entries, by a warp: lane r
// < 6 holds row r of [H | -g] and ends with x_r (Gauss-Jordan; H is symmetric
// positive definite, so its pivots need no exchange and are all positive: false
// otherwise).
__device__ __forceinline__ bool solve6(const double *Hu, const double *g, int lane, double &x)
{
    const int r = lane < 6 ? lane : 5;
    double m[7];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const int i = r < c ? r : c, j = r < c ? c : r;
        m[c] = Hu[6 * i - i * (i - 1) / 2 + (j - i)];
    }
    m[6] = -g[r];
    const double ridge = 1e-9 / 6.0 * (Hu[0] + Hu[6] + Hu[11] + Hu[15] + Hu[18] + Hu[20]);
#pragma unroll
    for (int c = 0; c < 6; ++c)
        if (r == c) m[c] += ridge;
    bool ok = true;
    x = 0.0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double row[7];
#pragma unroll
        for (int c = 0; c < 7; ++c)
            if (c >= j) row[c] = __shfl_sync(0xffffffffu, m[c], j);
        ok = ok && row[j] > 0.0 && row[j] < INFINITY;
        const double inv = recip(row[j]);
        const double f = r == j ? 0.0 : m[j] * inv;
        if (r == j) x = inv;
#pragma unroll
        for (int c = 0; c < 7; ++c)
            if (c > j) m[c] = fma(-f, row[c], m[c]);
    }
    x *= m[6];
    return ok;
}

__global__ void __launch_bounds__(PNP_THREADS) k_refine_pnp(PnpArgs a)
{
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    constexpr int NW = PNP_THREADS / 32;
    __shared__ double s_red[NW][PNP_ACC];
    __shared__ double s_tot[PNP_ACC];                    // the last pass's totals
    __shared__ double s_pose[12], s_trial[PNP_HALVINGS][12], s_delta[6];
    __shared__ int s_ok;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // pairs go round the blocks, so that a block's first warps hold its share
    const int first = blockIdx.x + gridDim.x * threadIdx.x, stride = gridDim.x * PNP_THREADS;
    int turn = 0;                                        // which half of the partial sums a pass writes
    double *c_now = a.c, *c_trial = a.c + a.n;           // exchanged when a step is taken

    // back-projection of every pair with the rendered depth
    for (int i = first; i < a.n; i += stride) {
        const float4 p = a.pairs[i];
        double4 X = make_double4(0.0, 0.0, 0.0, 0.0);
        const double sx = (double)p.x - 0.5, sy = (double)p.y - 0.5;
        if (isfinite(sx) && isfinite(sy) && isfinite((double)p.z) && isfinite((double)p.w)) {
            const double fx0 = floor(sx), fy0 = floor(sy);
            if (fx0 >= 0.0 && fy0 >= 0.0 && fx0 + 1.0 < (double)a.width && fy0 + 1.0 < (double)a.height) {
                const int x0 = (int)fx0, y0 = (int)fy0;
                const double wx = sx - fx0, wy = sy - fy0;
                const int64_t o = (int64_t)y0 * a.width + x0;
                const double D = (1 - wy) * ((1 - wx) * a.depth[o] + wx * a.depth[o + 1]) +
                                 wy * ((1 - wx) * a.depth[o + a.width] + wx * a.depth[o + a.width + 1]);
                const double A = (1 - wy) * ((1 - wx) * a.alpha[o] + wx * a.alpha[o + 1]) +
                                 wy * ((1 - wx) * a.alpha[o + a.width] + wx * a.alpha[o + a.width + 1]);
                if (A >= a.alpha_min) {
                    const double z = D / A;
                    const double c[3] = {z * ((double)p.x - a.cx) / a.fx - a.tr[0],
                                         z * ((double)p.y - a.cy) / a.fy - a.tr[1], z - a.tr[2]};
                    X.x = a.Rr[0] * c[0] + a.Rr[3] * c[1] + a.Rr[6] * c[2];
                    X.y = a.Rr[1] * c[0] + a.Rr[4] * c[1] + a.Rr[7] * c[2];
                    X.z = a.Rr[2] * c[0] + a.Rr[5] * c[1] + a.Rr[8] * c[2];
                    X.w = 1.0;
                }
            }
        }
        a.X[i] = X;                                      // read back by this block only
        a.c[i] = 0.0;
    }

    // The grid's totals of this lane's warp sum v (lane j: entry j) into s_tot,
    // the same on every block: blocks' sums through a.part, one grid barrier.
    auto grid_totals = [&](double v) {
        s_red[warp][lane] = v;
        __syncthreads();
        double *part = a.part + (int64_t)turn * gridDim.x * PNP_ACC;
        turn ^= 1;                                       // a block may still read these while the next pass writes
        if (warp == 0) {
            const double t = (s_red[0][lane] + s_red[1][lane]) + (s_red[2][lane] + s_red[3][lane]);
            __stcg(part + (int64_t)blockIdx.x * PNP_ACC + lane, t);
        }
        grid.sync();
        // four running sums of the warp's quarter of the blocks, all loads of a round in flight
        double t4[4] = {0.0, 0.0, 0.0, 0.0};
        for (int b = warp; b < (int)gridDim.x; b += 8 * NW) {
            double x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                x[k] = b + k * NW < (int)gridDim.x ? __ldcg(part + (int64_t)(b + k * NW) * PNP_ACC + lane) : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) t4[k & 3] += x[k];
        }
        s_red[warp][lane] = (t4[0] + t4[1]) + (t4[2] + t4[3]);
        __syncthreads();
        static_assert(NW == 4, "sums of four warps");
        if (warp == 0) s_tot[lane] = (s_red[0][lane] + s_red[1][lane]) + (s_red[2][lane] + s_red[3][lane]);
        __syncthreads();
    };
    // normal equations, cost and squared error at pose W (shared memory)
    auto evaluate = [&](const double *W) {
        double acc[PNP_ACC];
#pragma unroll
        for (int j = 0; j < PNP_ACC; ++j) acc[j] = 0.0;
        // a warp without pairs adds nothing (its FP64 instructions would take the same time)
        double v = 0.0;
        if (__any_sync(0xffffffffu, first < a.n)) {
            for (int i = first; i < a.n; i += stride) {
                const double c = pnp_add(a, W, a.X[i], a.pairs[i], acc);
                acc[PA_CHANGE] += c - c_now[i];
                c_trial[i] = c;
            }
            v = warp_sums<PNP_ACC>(acc, lane);
        }
        grid_totals(v);
    };

    if (threadIdx.x < 12) s_pose[threadIdx.x] = a.W0[threadIdx.x];
    __syncthreads();
    evaluate(s_pose);
    auto taken = [&]() {
        double *const t = c_now;
        c_now = c_trial;
        c_trial = t;
    };
    taken();
    const double n_used = s_tot[PA_USED];
    double cost = s_tot[PA_COST], sq = s_tot[PA_SQ], cnt = s_tot[PA_CNT];
    int it = 0;
    if (n_used >= 3.0) {
        for (; it < a.max_iters; ++it) {
            if (warp == 0) {
                double x;
                const bool ok = solve6(s_tot, s_tot + PA_G, lane, x);
                if (lane < 6) s_delta[lane] = x;
                if (lane == 0) s_ok = ok;
                __syncwarp();
                if (lane < 12) s_trial[0][lane] = update_entry(s_pose, s_delta, 1.0, lane);
            }
            __syncthreads();
            if (!s_ok) break;
            evaluate(s_trial[0]);
            double step = 1.0;
            int take = 0;
            if (!(s_tot[PA_CHANGE] < 0.0)) {
                // the halved steps, all in one pass
                for (int k = threadIdx.x; k < 12 * PNP_HALVINGS; k += PNP_THREADS) {
                    const int h = k / 12;
                    s_trial[h][k - 12 * h] = update_entry(s_pose, s_delta, 1.0 / (double)(2 << h), k - 12 * h);
                }
                __syncthreads();
                // threads 0..63 evaluate the first five, threads 64..127 the others, on the same pairs
                constexpr int HALF = PNP_HALVINGS / 2;
                const int h0 = threadIdx.x < PNP_THREADS / 2 ? 0 : HALF;
                double c[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) c[k] = 0.0;
                for (int i = blockIdx.x + gridDim.x * (threadIdx.x & (PNP_THREADS / 2 - 1)); i < a.n; i += stride / 2) {
                    const double4 X = a.X[i];
                    const float4 q = a.pairs[i];
                    if (X.w == 0.0) continue;
                    const double now = c_now[i];
#pragma unroll
                    for (int k = 0; k < HALF; ++k) {
                        double px, py, iz, ru, rv, e2, w;
                        c[k] += (pnp_residual(a, s_trial[h0 + k], X, q, px, py, iz, ru, rv, e2) ? huber(e2, a.huber, w) : 0.0) - now;
                    }
                }
                // lanes 4 k .. 4 k + 3 of a warp hold its sum k; entry 8 half + k of the pass
                const double cs = __shfl_sync(0xffffffffu, warp_sums<8>(c, lane), (4 * lane) & 31);
                grid_totals(lane >= 8 && lane < 16 ? (h0 ? cs : 0.0) : lane < 8 ? (h0 ? 0.0 : cs) : 0.0);
                auto change = [&](int h) { return s_tot[h < HALF ? h : 8 + h - HALF]; };
                for (take = 0; take < PNP_HALVINGS && !(change(take) < 0.0); ++take) {}
                if (take == PNP_HALVINGS) break;         // no step lowers the cost: converged
                step = 1.0 / (double)(2 << take);
                __syncthreads();                         // s_tot is read before the pass below writes it
                evaluate(s_trial[take]);
            }
            taken();
            cost = s_tot[PA_COST];
            sq = s_tot[PA_SQ];
            cnt = s_tot[PA_CNT];
            if (threadIdx.x < 12) s_pose[threadIdx.x] = s_trial[take][threadIdx.x];
            // read before the barrier: after it the first warp may write the next step
            // already, and a warp that judged by that one could leave alone
            double dmax = 0.0;
            for (int j = 0; j < 6; ++j) dmax = fmax(dmax, fabs(step * s_delta[j]));
            __syncthreads();
            if (dmax < a.tol) {
                ++it;
                break;
            }
        }
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int r = 0; r < 3; ++r) {
            for (int c = 0; c < 3; ++c) a.out[4 * r + c] = s_pose[3 * r + c];
            a.out[4 * r + 3] = s_pose[9 + r];
        }
        a.out[12] = a.out[13] = a.out[14] = 0.0;
        a.out[15] = 1.0;
        a.out[16] = cnt > 0.0 ? sqrt(sq / cnt) : 0.0;
        a.out[17] = cost;
        a.out[18] = n_used;
        a.out[19] = (double)it;
    }
}

cudaError_t launch_refine_pnp(const double *pose_render, const double *pose_init, double fx, double fy, double cx,
                              double cy, int width, int height, const float *depth, const float *alpha,
                              const float *pairs, int n, int max_iters, double huber, double alpha_min, double tol,
                              double *X_scratch, double *out, cudaStream_t st)
{
    PnpArgs a;
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c) {
            a.Rr[3 * r + c] = pose_render[4 * r + c];
            a.W0[3 * r + c] = pose_init[4 * r + c];
        }
        a.tr[r] = pose_render[4 * r + 3];
        a.W0[9 + r] = pose_init[4 * r + 3];
    }
    a.fx = fx; a.fy = fy; a.cx = cx; a.cy = cy;
    a.width = width; a.height = height; a.n = n; a.max_iters = max_iters;
    a.huber = huber; a.alpha_min = alpha_min; a.tol = tol;
    a.depth = depth; a.alpha = alpha;
    a.pairs = reinterpret_cast<const float4 *>(pairs);
    a.X = reinterpret_cast<double4 *>(X_scratch);
    a.out = out;
    // at most one block per SM (all resident: the launch is cooperative), of a warp's
    // worth of pairs or more
    int dev = 0, n_sm = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(n_sm, ceil_div(n, 32)));
    a.c = X_scratch + 4 * (int64_t)n;
    a.part = a.c + 2 * (int64_t)n;
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel((const void *)k_refine_pnp, dim3(nb), dim3(PNP_THREADS), args, 0, st);
    return e;
}

}  // namespace reloc
