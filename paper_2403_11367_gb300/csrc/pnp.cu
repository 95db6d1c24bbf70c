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
// FP64 instruction holds the SM's pipe for some 15 clocks.  So the pairs are
// spread two warps to an SM over one cooperative launch, and what counts is the
// number of passes over the pairs, the barriers between them and the FP64
// instructions of a reduction:
//   - one pass per iteration: the trial pose is evaluated with its normal
//     equations, so an accepted step has them already (and the final pose its
//     cost and squared error);
//   - one grid barrier per pass: every block adds all blocks' partial sums, in
//     the same order, and solves the system for itself, so nothing is handed
//     back from a leading block;
//   - when the full step does not lower the cost (every solve ends there: the
//     cost is flat to rounding at the minimum) the ten halved steps are
//     evaluated in one pass, not one by one;
//   - a warp sums its 32 accumulators by recursive halving (31 additions, lane
//     j left with total j) instead of 28 butterflies of five.
// Some 7,000 pairs on the driving street: 529 us a call with one block per 256
// pairs, five barriers and two passes an iteration, 241 us so.
#include <algorithm>

#include <cooperative_groups.h>

#include "internal.cuh"

namespace reloc {

constexpr int PNP_MAX_THREADS = 128;
constexpr int PNP_HALVINGS = 10;         // backtracking: the step is halved at most this often
// accumulators of a pass: upper H (21), g (6), Huber cost, pairs with a point,
// squared error and count of the pairs in front of the camera
enum { PA_G = 21, PA_COST = 27, PA_USED = 28, PA_SQ = 29, PA_CNT = 30, PNP_ACC = 32 };

struct PnpArgs {
    double Rr[9], tr[3];                 // render pose (world -> camera)
    double W0[12];                       // initial pose: R row-major, then t
    double fx, fy, cx, cy;
    int width, height, n, max_iters;
    double huber, alpha_min, tol;
    const float *depth, *alpha;
    const float4 *pairs;
    double4 *X;                          // scratch [n]: world point, w = 1 if used
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

__device__ __forceinline__ double huber_rho(double e, double k) { return e <= k ? 0.5 * e * e : k * (e - 0.5 * k); }

// One pair's residual at pose W (R row-major, then t): false behind the camera.
__device__ __forceinline__ bool pnp_residual(const PnpArgs &a, const double *W, const double4 &X, const float4 &q,
                                             double &px, double &py, double &iz, double &ru, double &rv, double &e2)
{
    px = W[0] * X.x + W[1] * X.y + W[2] * X.z + W[9];
    py = W[3] * X.x + W[4] * X.y + W[5] * X.z + W[10];
    const double pz = W[6] * X.x + W[7] * X.y + W[8] * X.z + W[11];
    if (pz <= 1e-6) return false;
    iz = 1.0 / pz;
    ru = a.fx * px * iz + a.cx - (double)q.z;
    rv = a.fy * py * iz + a.cy - (double)q.w;
    e2 = ru * ru + rv * rv;
    return true;
}

// Adds one pair's normal equations, cost and squared error at pose W.  The
// Jacobian rows are Ju = (u0, 0, u2, u3, u4, u5), Jv = (0, v1, v2, v3, v4, v5).
__device__ __forceinline__ void pnp_add(const PnpArgs &a, const double *W, const double4 &X, const float4 &q,
                                        double (&acc)[PNP_ACC])
{
    if (X.w == 0.0) return;
    acc[PA_USED] += 1.0;
    double px, py, iz, ru, rv, e2;
    if (!pnp_residual(a, W, X, q, px, py, iz, ru, rv, e2)) return;
    const double e = sqrt(e2);
    acc[PA_COST] += huber_rho(e, a.huber);
    acc[PA_SQ] += e * e;
    acc[PA_CNT] += 1.0;
    const double w = e <= a.huber ? 1.0 : a.huber / e;
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
}

// W' = [Exp(phi) R | Exp(phi) t + rho] for delta = (rho, phi) scaled by s.
__device__ void apply_update(const double *W, const double *delta, double s, double *Wn)
{
    const double rho[3] = {s * delta[0], s * delta[1], s * delta[2]};
    const double ph[3] = {s * delta[3], s * delta[4], s * delta[5]};
    const double th2 = ph[0] * ph[0] + ph[1] * ph[1] + ph[2] * ph[2], th = sqrt(th2);
    double A, B;                                   // Exp = I + A K + B K^2, K = [phi]x
    if (th < 1e-8) {
        A = 1.0 - th2 / 6.0;
        B = 0.5 - th2 / 24.0;
    } else {
        double sn, cs;
        sincos(th, &sn, &cs);
        A = sn / th;
        B = (1.0 - cs) / th2;
    }
    const double K[9] = {0.0, -ph[2], ph[1], ph[2], 0.0, -ph[0], -ph[1], ph[0], 0.0};
    double E[9];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            double k2 = 0.0;
            for (int m = 0; m < 3; ++m) k2 += K[3 * r + m] * K[3 * m + c];
            E[3 * r + c] = (r == c ? 1.0 : 0.0) + A * K[3 * r + c] + B * k2;
        }
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c)
            Wn[3 * r + c] = E[3 * r] * W[c] + E[3 * r + 1] * W[3 + c] + E[3 * r + 2] * W[6 + c];
        Wn[9 + r] = E[3 * r] * W[9] + E[3 * r + 1] * W[10] + E[3 * r + 2] * W[11] + rho[r];
    }
}

// Solve (H + 1e-9 tr(H)/6 I) x = -g by Cholesky; H given as 21 upper entries.
// Unrolled into registers, with one reciprocal per pivot.
__device__ __forceinline__ bool solve6(const double *Hu, const double *g, double (&x)[6])
{
    double H[6][6];
    {
        int k = 0;
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int c = r; c < 6; ++c) H[c][r] = Hu[k++];
    }
    const double ridge = 1e-9 * (H[0][0] + H[1][1] + H[2][2] + H[3][3] + H[4][4] + H[5][5]) / 6.0;
    double il[6];
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double d = H[j][j] + ridge;
#pragma unroll
        for (int m = 0; m < 6; ++m)
            if (m < j) d -= H[j][m] * H[j][m];
        ok = ok && d > 0.0;
        il[j] = 1.0 / sqrt(d);
#pragma unroll
        for (int i = 0; i < 6; ++i)
            if (i > j) {
                double s = H[i][j];
#pragma unroll
                for (int m = 0; m < 6; ++m)
                    if (m < j) s -= H[i][m] * H[j][m];
                H[i][j] = s * il[j];
            }
    }
    double y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        double s = -g[i];
#pragma unroll
        for (int m = 0; m < 6; ++m)
            if (m < i) s -= H[i][m] * y[m];
        y[i] = s * il[i];
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        double s = y[i];
#pragma unroll
        for (int m = 0; m < 6; ++m)
            if (m > i) s -= H[m][i] * x[m];
        x[i] = s * il[i];
    }
    return ok;
}

__global__ void __launch_bounds__(PNP_MAX_THREADS) k_refine_pnp(PnpArgs a)
{
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    constexpr int MAX_WARPS = PNP_MAX_THREADS / 32;
    __shared__ double s_red[MAX_WARPS][PNP_ACC];
    __shared__ double s_tot[PNP_ACC];                    // the last pass's totals
    __shared__ double s_pose[12], s_trial[PNP_HALVINGS][12], s_delta[6];
    __shared__ int s_ok;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    int turn = 0;                                        // which half of the partial sums a pass writes

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
        a.X[i] = X;                                      // read back by this thread only
    }

    // The grid's totals of this lane's warp sum v (lane j: entry j) into s_tot,
    // the same on every block: blocks' sums through a.part, one grid barrier.
    auto grid_totals = [&](double v) {
        s_red[warp][lane] = v;
        __syncthreads();
        double *part = a.part + (int64_t)turn * gridDim.x * PNP_ACC;
        turn ^= 1;                                       // a block may still read these while the next pass writes
        if (warp == 0) {
            double t = s_red[0][lane];
            for (int w = 1; w < n_warps; ++w) t += s_red[w][lane];
            __stcg(part + (int64_t)blockIdx.x * PNP_ACC + lane, t);
        }
        grid.sync();
        double t = 0.0;
        int b = warp;
        for (; b + 7 * n_warps < (int)gridDim.x; b += 8 * n_warps) {
            double x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = __ldcg(part + (int64_t)(b + k * n_warps) * PNP_ACC + lane);
#pragma unroll
            for (int k = 0; k < 8; ++k) t += x[k];
        }
        for (; b < (int)gridDim.x; b += n_warps) t += __ldcg(part + (int64_t)b * PNP_ACC + lane);
        s_red[warp][lane] = t;
        __syncthreads();
        if (warp == 0) {
            t = s_red[0][lane];
            for (int w = 1; w < n_warps; ++w) t += s_red[w][lane];
            s_tot[lane] = t;
        }
        __syncthreads();
    };
    // normal equations, cost and squared error at pose W (shared memory)
    auto evaluate = [&](const double *W) {
        double acc[PNP_ACC];
#pragma unroll
        for (int j = 0; j < PNP_ACC; ++j) acc[j] = 0.0;
        for (int i = first; i < a.n; i += stride) pnp_add(a, W, a.X[i], a.pairs[i], acc);
        grid_totals(warp_sums<PNP_ACC>(acc, lane));
    };

    if (threadIdx.x < 12) s_pose[threadIdx.x] = a.W0[threadIdx.x];
    __syncthreads();
    evaluate(s_pose);
    const double n_used = s_tot[PA_USED];
    double cost = s_tot[PA_COST], sq = s_tot[PA_SQ], cnt = s_tot[PA_CNT];
    int it = 0;
    if (n_used >= 3.0) {
        for (; it < a.max_iters; ++it) {
            if (threadIdx.x == 0) {
                double d[6];
                s_ok = solve6(s_tot, s_tot + PA_G, d);
                for (int j = 0; j < 6; ++j) s_delta[j] = d[j];
                apply_update(s_pose, d, 1.0, s_trial[0]);
            }
            __syncthreads();
            if (!s_ok) break;
            evaluate(s_trial[0]);
            double step = 1.0;
            int take = 0;
            if (!(s_tot[PA_COST] < cost)) {
                // the halved steps, all in one pass
                if (threadIdx.x < PNP_HALVINGS)
                    apply_update(s_pose, s_delta, 1.0 / (double)(2 << threadIdx.x), s_trial[threadIdx.x]);
                __syncthreads();
                double c[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) c[k] = 0.0;
                for (int i = first; i < a.n; i += stride) {
                    const double4 X = a.X[i];
                    const float4 q = a.pairs[i];
                    if (X.w == 0.0) continue;
#pragma unroll
                    for (int k = 0; k < PNP_HALVINGS; ++k) {
                        double px, py, iz, ru, rv, e2;
                        if (pnp_residual(a, s_trial[k], X, q, px, py, iz, ru, rv, e2)) c[k] += huber_rho(sqrt(e2), a.huber);
                    }
                }
                grid_totals(warp_sums<16>(c, lane));     // lanes 2 k and 2 k + 1: step k
                for (take = 0; take < PNP_HALVINGS && !(s_tot[2 * take] < cost); ++take) {}
                if (take == PNP_HALVINGS) break;         // no step lowers the cost: converged
                step = 1.0 / (double)(2 << take);
                __syncthreads();                         // s_tot is read before the pass below writes it
                evaluate(s_trial[take]);
            }
            cost = s_tot[PA_COST];
            sq = s_tot[PA_SQ];
            cnt = s_tot[PA_CNT];
            if (threadIdx.x < 12) s_pose[threadIdx.x] = s_trial[take][threadIdx.x];
            __syncthreads();
            double dmax = 0.0;
            for (int j = 0; j < 6; ++j) dmax = fmax(dmax, fabs(step * s_delta[j]));
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
    // at most one block per SM (all resident: the launch is cooperative), of two
    // warps while that covers the pairs one each, of four beyond
    int dev = 0, n_sm = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int nt = n <= 64 * n_sm ? 64 : PNP_MAX_THREADS;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(n_sm, ceil_div(n, nt)));
    a.part = X_scratch + 4 * (int64_t)n;
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel((const void *)k_refine_pnp, dim3(nb), dim3(nt), args, 0, st);
    return e;
}

}  // namespace reloc
