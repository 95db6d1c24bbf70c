// cnn.cu -- elementwise and layout kernels of the learned candidate proposal
// (the dense contractions run in gemm.cu).
//
// The proposal network ranks the candidates of the relocalization grid from a
// low-resolution view of the query and of the coarse-pose render, so that only
// the most likely candidates are rendered and scored (the full sweep of
// Sec. III-C.1 stays as the fallback).  Activations are NHWC BF16; every
// convolution is 3x3, stride 2, padding 1, lowered to a GEMM by im2col with
// column index k = (ky * 3 + kx) * C_in + c_in (zero-padded to a multiple of 64).
#include "internal.cuh"

namespace reloc {

// f x f box average of the RGB mean (gray) of planar [3][H][W] images into NHWC
// [n][H / f][W / f][2] BF16 inputs: channel 0 from query j, channel 1 from render j.
// A thread sums one output in a fixed order (rows, columns, r + g + b).  One launch
// for GRAY_PAIRS queries and renders; bound by reading them (406 MB for 32 driving
// queries, 60 us).  An image a launch and a value a load kept 33 blocks of 256
// threads waiting for one row after the other: 64 launches of 11 us, 62 us
// now.  VEC: f a multiple of 4 and rows on 16 bytes, so four columns a load.
template <bool VEC>
__global__ void __launch_bounds__(256)
k_downsample_gray(GrayQueries q, const float *__restrict__ render, int H, int W, int f, __nv_bfloat16 *__restrict__ out)
{
    const int Ho = H / f, Wo = W / f;
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= Ho * Wo) return;
    const int j = blockIdx.y >> 1, ch = blockIdx.y & 1;
    const int oy = i / Wo, ox = i % Wo;
    const int64_t HW = (int64_t)H * W;
    const float *img = ch ? render + 3 * HW * j : q.img[j];
    float s = 0.f;
    if (VEC) {
#pragma unroll 2
        for (int y = oy * f; y < oy * f + f; ++y)
#pragma unroll 2
            for (int x = ox * f; x < ox * f + f; x += 4) {
                const float *p = img + (int64_t)y * W + x;
                const float4 r = *reinterpret_cast<const float4 *>(p), g = *reinterpret_cast<const float4 *>(p + HW),
                             b = *reinterpret_cast<const float4 *>(p + 2 * HW);
                s += r.x + g.x + b.x;
                s += r.y + g.y + b.y;
                s += r.z + g.z + b.z;
                s += r.w + g.w + b.w;
            }
    } else {
        for (int y = oy * f; y < oy * f + f; ++y)
            for (int x = ox * f; x < ox * f + f; ++x) {
                const int64_t p = (int64_t)y * W + x;
                s += img[p] + img[HW + p] + img[2 * HW + p];
            }
    }
    out[((int64_t)j * Ho * Wo + i) * 2 + ch] = __float2bfloat16_rn(s / (3.f * f * f));
}

cudaError_t launch_downsample_gray(const GrayQueries &q, const float *render, int n, int H, int W, int f,
                                   __nv_bfloat16 *out, cudaStream_t st)
{
    bool vec = f % 4 == 0 && W % 4 == 0 && ((uintptr_t)render & 15) == 0;
    for (int j = 0; j < n; ++j) vec = vec && ((uintptr_t)q.img[j] & 15) == 0;
    const dim3 grid((unsigned)(((H / f) * (W / f) + 255) / 256), (unsigned)(2 * n));
    if (vec)
        k_downsample_gray<true><<<grid, 256, 0, st>>>(q, render, H, W, f, out);
    else
        k_downsample_gray<false><<<grid, 256, 0, st>>>(q, render, H, W, f, out);
    return cudaGetLastError();
}

// im2col for a 3x3 / stride 2 / pad 1 convolution: X [B][H][W][C] ->
// col [B*Ho*Wo][Kp], zero beyond K = 9 C.  A thread writes eight columns, 16
// bytes: eight channels of one tap, or for the two-channel input four taps, each one
// 4-byte load (PAIR) or, of a caller's buffer off 4 bytes, two 2-byte loads.
// Bound by its writes (211 MB for the five layers at batch 256; one value a
// thread took 650 us there).
constexpr int COL_THREADS = 256;
template <bool PAIR>
__global__ void __launch_bounds__(COL_THREADS)
k_im2col(const __nv_bfloat16 *__restrict__ x, int M, int H, int W, int C, int Ho, int Wo, int Kp,
         __nv_bfloat16 *__restrict__ col)
{
    const int G = Kp / 8, rows = COL_THREADS / G;         // groups of a row, rows of a block
    const int r = threadIdx.x / G, g = threadIdx.x - r * G;
    const int64_t row64 = (int64_t)blockIdx.x * rows + r;
    if (r >= rows || row64 >= M) return;
    const int row = (int)row64;
    const int ox = row % Wo, t = row / Wo, oy = t % Ho, b = t / Ho;
    const __nv_bfloat16 *xb = x + (int64_t)b * H * W * C;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (C == 2) {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int tap = 4 * g + j, y = 2 * oy - 1 + tap / 3, xx = 2 * ox - 1 + tap % 3;
            if (tap < 9 && y >= 0 && y < H && xx >= 0 && xx < W) {
                const __nv_bfloat16 *p = xb + ((int64_t)y * W + xx) * 2;
                w[j] = PAIR ? *reinterpret_cast<const uint32_t *>(p)
                            : (uint32_t)__bfloat16_as_ushort(p[0]) | (uint32_t)__bfloat16_as_ushort(p[1]) << 16;
            }
        }
        v = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
        const int k = 8 * g, tap = k / C, ci = k - tap * C;
        const int y = 2 * oy - 1 + tap / 3, xx = 2 * ox - 1 + tap % 3;
        if (tap < 9 && y >= 0 && y < H && xx >= 0 && xx < W)
            v = *reinterpret_cast<const uint4 *>(xb + ((int64_t)y * W + xx) * C + ci);
    }
    *reinterpret_cast<uint4 *>(col + row64 * Kp + 8 * g) = v;
}

// C 2 or a multiple of 8; Kp a multiple of 8, at most 8 * 256; x on 2 (C = 2) or 16 bytes.
cudaError_t launch_im2col(const __nv_bfloat16 *x, int B, int H, int W, int C, int Ho, int Wo, int Kp,
                          __nv_bfloat16 *col, cudaStream_t st)
{
    if ((C != 2 && (C % 8 || ((uintptr_t)x & 15))) || Kp % 8 || Kp / 8 > COL_THREADS) return cudaErrorInvalidValue;
    const int M = B * Ho * Wo;
    const unsigned grid = (unsigned)ceil_div(M, COL_THREADS / (Kp / 8));
    if (((uintptr_t)x & 3) == 0) k_im2col<true><<<grid, COL_THREADS, 0, st>>>(x, M, H, W, C, Ho, Wo, Kp, col);
    else k_im2col<false><<<grid, COL_THREADS, 0, st>>>(x, M, H, W, C, Ho, Wo, Kp, col);
    return cudaGetLastError();
}

// A backward signal carried as two BF16 terms: out [M][2N] holds hi =
// bf16(x) in columns 0..N-1 and lo = bf16(x - hi) in N..2N-1, so hi + lo
// keeps ~16 significant bits of x and the GEMMs that contract it (over 2N
// columns, or 2M rows stacked) accumulate both in FP32.
__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 &hi, __nv_bfloat16 &lo)
{
    hi = __float2bfloat16_rn(x);
    lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// Gradient through a ReLU at the stored activations y [M][N], split into hi | lo,
// with the bias gradient's per-block column sums (of hi + lo) in part[block][N].
// The incoming gradient is d [M][N] (C2I false), or the col2im of dcol (true):
// row p = (b, y, x) of the layer's input sums, over the (ky, kx) in order whose
// output position (oy, ox) with y = 2 oy - 1 + ky, x = 2 ox - 1 + kx lies in the
// output, dcol[(b, oy, ox)][(ky, kx, c)].  A thread takes four columns of every
// `step`-th row, so rows are read and written whole, the col2im's result never
// goes to memory, and the sums cost no pass of their own (as separate kernels of
// one value a thread, and a block per column for the sums: 254 + 148 + 733 us of
// a step of batch 256).
struct Col2Im {
    int H, W, Ho, Wo, Kp;
};
constexpr int RB_THREADS = 256;
template <bool C2I>
__global__ void __launch_bounds__(RB_THREADS)
k_relu_back(const float *__restrict__ d, Col2Im g, const __nv_bfloat16 *__restrict__ y, int M, int N,
            __nv_bfloat16 *__restrict__ out, float *__restrict__ part)
{
    extern __shared__ float4 s_sum[];                     // [rows of a block][N / 4]
    const int NG = N / 4, rows = RB_THREADS / NG > 0 ? RB_THREADS / NG : 1;
    const int gpt = NG > RB_THREADS ? NG / RB_THREADS : 1;   // column groups a thread walks (N a multiple of 1024 then)
    const int r = threadIdx.x / (NG < RB_THREADS ? NG : RB_THREADS);
    const int c0 = threadIdx.x - r * NG;
    for (int q = 0; q < gpt; ++q) {
        const int c = (NG < RB_THREADS ? c0 : (int)threadIdx.x + q * RB_THREADS) * 4;
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows)
            for (int64_t row = (int64_t)blockIdx.x * rows + r; row < M; row += (int64_t)gridDim.x * rows) {
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                if (C2I) {
                    const int p = (int)row, px = p % g.W, t = p / g.W, py = t % g.H, b = t / g.H;
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        const int ty = py + 1 - ky, oy = ty >> 1;
                        if ((ty & 1) || oy < 0 || oy >= g.Ho) continue;
#pragma unroll
                        for (int kx = 0; kx < 3; ++kx) {
                            const int tx = px + 1 - kx, ox = tx >> 1;
                            if ((tx & 1) || ox < 0 || ox >= g.Wo) continue;
                            const float4 v = __ldg(reinterpret_cast<const float4 *>(
                                d + (((int64_t)b * g.Ho + oy) * g.Wo + ox) * g.Kp + (ky * 3 + kx) * N + c));
                            x.x += v.x; x.y += v.y; x.z += v.z; x.w += v.w;
                        }
                    }
                } else {
                    x = __ldg(reinterpret_cast<const float4 *>(d + row * N + c));
                }
                const uint2 yb = __ldg(reinterpret_cast<const uint2 *>(y + row * N + c));
                const __nv_bfloat162 y01 = *reinterpret_cast<const __nv_bfloat162 *>(&yb.x);
                const __nv_bfloat162 y23 = *reinterpret_cast<const __nv_bfloat162 *>(&yb.y);
                __nv_bfloat162 h[2], l[2];
                split_bf16((float)y01.x > 0.f ? x.x : 0.f, h[0].x, l[0].x);
                split_bf16((float)y01.y > 0.f ? x.y : 0.f, h[0].y, l[0].y);
                split_bf16((float)y23.x > 0.f ? x.z : 0.f, h[1].x, l[1].x);
                split_bf16((float)y23.y > 0.f ? x.w : 0.f, h[1].y, l[1].y);
                sum.x += (float)h[0].x + (float)l[0].x;
                sum.y += (float)h[0].y + (float)l[0].y;
                sum.z += (float)h[1].x + (float)l[1].x;
                sum.w += (float)h[1].y + (float)l[1].y;
                __nv_bfloat16 *o = out + row * 2 * N + c;
                *reinterpret_cast<uint2 *>(o) = *reinterpret_cast<const uint2 *>(h);
                *reinterpret_cast<uint2 *>(o + N) = *reinterpret_cast<const uint2 *>(l);
            }
        if (rows == 1) {
            // (widths between half a block's threads and all of them leave some without a row)
            if (r == 0) *reinterpret_cast<float4 *>(part + (int64_t)blockIdx.x * N + c) = sum;
            continue;
        }
        if (r < rows) s_sum[r * NG + c / 4] = sum;
        __syncthreads();
        if (r == 0) {
            for (int k = 1; k < rows; ++k) {
                const float4 v = s_sum[k * NG + c / 4];
                sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
            }
            *reinterpret_cast<float4 *>(part + (int64_t)blockIdx.x * N + c) = sum;
        }
    }
}

// db[c] = sum of part[0 .. n_part)[c], in a fixed order: eight runs a column.
__global__ void __launch_bounds__(256) k_colsum_final(const float *__restrict__ part, int n_part, int N, float *__restrict__ db)
{
    __shared__ float s[8][32];
    const int c = blockIdx.x * 32 + (threadIdx.x & 31), run = threadIdx.x >> 5;
    float a = 0.f;
    if (c < N)
        for (int k = run; k < n_part; k += 8) a += part[(int64_t)k * N + c];
    s[run][threadIdx.x & 31] = a;
    __syncthreads();
    if (run == 0 && c < N) {
        for (int k = 1; k < 8; ++k) a += s[k][threadIdx.x];
        db[c] = a;
    }
}

// ReLU backward into out [M][2N] (hi | lo) and the bias gradient db [N].  d
// [M][N], or with Ho > 0 the next layer's dcol [B*Ho*Wo][Kp], M = B*H*W.  N a
// multiple of 4, and of 1024 above 1024.  part: RELU_BACK_BLOCKS * N floats.
cudaError_t launch_relu_back(const float *d, int H, int W, int Ho, int Wo, int Kp, const __nv_bfloat16 *y, int M, int N,
                             __nv_bfloat16 *out, float *part, float *db, cudaStream_t st)
{
    const int NG = N / 4;
    if (M <= 0 || N % 4 || (NG > RB_THREADS && NG % RB_THREADS)) return cudaErrorInvalidValue;
    const int rows = NG < RB_THREADS ? RB_THREADS / NG : 1;
    const int blocks = (int)min64(ceil_div(M, rows), RELU_BACK_BLOCKS);
    const size_t smem = rows > 1 ? sizeof(float4) * rows * NG : 0;
    const Col2Im g{H, W, Ho, Wo, Kp};
    if (Ho > 0) k_relu_back<true><<<blocks, RB_THREADS, smem, st>>>(d, g, y, M, N, out, part);
    else k_relu_back<false><<<blocks, RB_THREADS, smem, st>>>(d, g, y, M, N, out, part);
    k_colsum_final<<<(unsigned)ceil_div(N, 32), 256, 0, st>>>(part, blocks, N, db);
    return cudaGetLastError();
}

// db[c] = sum over the R rows of the split signal d [R][2 Cc] (hi + lo), FP32
// (the logits' few rows and columns).
__global__ void k_colsum(const __nv_bfloat16 *__restrict__ d, int R, int Cc, float *__restrict__ db)
{
    __shared__ float s[256];
    const int c = blockIdx.x;
    float a = 0.f;
    for (int r = threadIdx.x; r < R; r += 256)
        a += (float)d[(int64_t)r * 2 * Cc + c] + (float)d[(int64_t)r * 2 * Cc + Cc + c];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) db[c] = s[0];
}

cudaError_t launch_colsum(const __nv_bfloat16 *d, int R, int Cc, float *db, cudaStream_t st)
{
    k_colsum<<<Cc, 256, 0, st>>>(d, R, Cc, db);
    return cudaGetLastError();
}

// Softmax cross-entropy rows: loss_rows[b], dl = (softmax - onehot) / B in
// FP32 and split into hi | lo BF16 terms (dlb [B][2C]).
__global__ void k_softmax_ce(const float *__restrict__ logits, const int32_t *__restrict__ labels, int B, int C,
                             float *__restrict__ loss_rows, float *__restrict__ dl, __nv_bfloat16 *__restrict__ dlb)
{
    const int b = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= B) return;
    const float *z = logits + (int64_t)b * C;
    float mx = -INFINITY;
    for (int c = lane; c < C; c += 32) mx = fmaxf(mx, z[c]);
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float se = 0.f;
    for (int c = lane; c < C; c += 32) se += expf(z[c] - mx);
    for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
    const int y = labels[b];
    for (int c = lane; c < C; c += 32) {
        const float p = expf(z[c] - mx) / se;
        const float g = (p - (c == y ? 1.f : 0.f)) / (float)B;
        dl[(int64_t)b * C + c] = g;
        split_bf16(g, dlb[(int64_t)b * 2 * C + c], dlb[(int64_t)b * 2 * C + C + c]);
    }
    if (lane == 0) loss_rows[b] = logf(se) + mx - z[y];
}

cudaError_t launch_softmax_ce(const float *logits, const int32_t *labels, int B, int C, float *loss_rows, float *dl,
                              __nv_bfloat16 *dlb, cudaStream_t st)
{
    k_softmax_ce<<<(unsigned)ceil_div(B, 8), 256, 0, st>>>(logits, labels, B, C, loss_rows, dl, dlb);
    return cudaGetLastError();
}

// Adam (Kingma and Ba): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// w -= lr * (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps), over all n
// parameters in one launch (two per tensor cost more in launches than the
// update takes).  Also refreshes the weights' BF16 copies: parameter i of
// [T.begin[k], T.end[k]) is T.bf[k] + i - T.begin[k] there (biases have none).
__global__ void k_adam(float *__restrict__ w, float *__restrict__ m, float *__restrict__ v, const float *__restrict__ g,
                       int64_t n, float lr, float b1, float b2, float eps, float c1, float c2, AdamTensors T,
                       __nv_bfloat16 *__restrict__ w_bf)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    int64_t at = -1;
#pragma unroll
    for (int k = 0; k < AdamTensors::N; ++k)
        if (i >= T.begin[k] && i < T.end[k]) at = T.bf[k] + (i - T.begin[k]);
    if (at >= 0) w_bf[at] = __float2bfloat16_rn(wi);
}

cudaError_t launch_adam(float *w, float *m, float *v, const float *g, int64_t n, float lr, float b1, float b2, float eps,
                        float c1, float c2, const AdamTensors &T, __nv_bfloat16 *w_bf, cudaStream_t st)
{
    k_adam<<<(unsigned)ceil_div(n, 256), 256, 0, st>>>(w, m, v, g, n, lr, b1, b2, eps, c1, c2, T, w_bf);
    return cudaGetLastError();
}

// FP32 -> BF16 copy.
__global__ void k_to_bf16(const float *__restrict__ a, int64_t n, __nv_bfloat16 *__restrict__ b)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = __float2bfloat16_rn(a[i]);
}

cudaError_t launch_to_bf16(const float *a, int64_t n, __nv_bfloat16 *b, cudaStream_t st)
{
    k_to_bf16<<<(unsigned)ceil_div(n, 256), 256, 0, st>>>(a, n, b);
    return cudaGetLastError();
}

// Top-k of each row of C logits (k <= 32), descending, ties by lower index;
// also the softmax margin p1 - p2.  One warp per row.
__global__ void k_topk(const float *__restrict__ logits, int B, int C, int k, int32_t *__restrict__ idx,
                       float *__restrict__ margin)
{
    const int b = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= B) return;
    const float *z = logits + (int64_t)b * C;
    float mx = -INFINITY;
    for (int c = lane; c < C; c += 32) mx = fmaxf(mx, z[c]);
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float se = 0.f;
    for (int c = lane; c < C; c += 32) se += expf(z[c] - mx);
    for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
    uint32_t taken[4] = {0, 0, 0, 0};     // up to 128 classes
    float p1 = 0.f, p2 = 0.f;
    for (int r = 0; r < k; ++r) {
        float best = -INFINITY;
        int bi = 0x7fffffff;
        for (int c = lane; c < C; c += 32)
            if (!((taken[c >> 5] >> (c & 31)) & 1u) && (z[c] > best || (z[c] == best && c < bi))) { best = z[c]; bi = c; }
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (bi >= C) break;
        taken[bi >> 5] |= 1u << (bi & 31);
        if (lane == 0) idx[(int64_t)b * k + r] = bi;
        if (r == 0) p1 = expf(best - mx) / se;
        if (r == 1) p2 = expf(best - mx) / se;
    }
    if (lane == 0) margin[b] = p1 - p2;
}

cudaError_t launch_topk(const float *logits, int B, int C, int k, int32_t *idx, float *margin, cudaStream_t st)
{
    if (C > 128 || k > 32 || k < 2) return cudaErrorInvalidValue;
    k_topk<<<(unsigned)ceil_div(B, 8), 256, 0, st>>>(logits, B, C, k, idx, margin);
    return cudaGetLastError();
}

}  // namespace reloc
