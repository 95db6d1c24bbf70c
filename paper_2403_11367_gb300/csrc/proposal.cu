// proposal.cu -- the learned candidate proposal: a small CNN that ranks the
// candidates of the relocalization grid from 176x47 gray views of the query
// and of the coarse-pose render, trained on the GPU with the kernels of
// gemm.cu (tcgen05 BF16 tensor cores, FP32 accumulation) and cnn.cu.
//
// Architecture (input NHWC [B][47][176][2]):
//   5 x { 3x3 conv, stride 2, pad 1, + bias, ReLU }: 2 -> 32 -> 64 -> 64 -> 128 -> 128
//   (spatial 47x176 -> 24x88 -> 12x44 -> 6x22 -> 3x11 -> 2x6)
//   flatten (NHWC order, 1536) -> FC 1024 + ReLU -> FC 64 (logits)
// Loss: softmax cross-entropy, mean over the batch; optimiser: Adam.
//
// Flat parameter layout (FP32, used for save/load and for checks): for each
// conv layer W[C_out][3][3][C_in] then b[C_out]; then FC1 W[1024][1536],
// b[1024]; FC2 W[64][1024], b[64] -- 1,916,960 values.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.cuh"

namespace reloc {

cudaError_t launch_downsample_gray(const GrayQueries &q, const float *render, int n, int H, int W, int f,
                                   __nv_bfloat16 *out, cudaStream_t st);
cudaError_t launch_im2col(const __nv_bfloat16 *x, int B, int H, int W, int C, int Ho, int Wo, int Kp,
                          __nv_bfloat16 *col, cudaStream_t st);
cudaError_t launch_relu_back(const float *d, int H, int W, int Ho, int Wo, int Kp, const __nv_bfloat16 *y, int M, int N,
                             __nv_bfloat16 *out, float *part, float *db, cudaStream_t st);
cudaError_t launch_colsum(const __nv_bfloat16 *d, int R, int Cc, float *db, cudaStream_t st);
cudaError_t launch_softmax_ce(const float *logits, const int32_t *labels, int B, int C, float *loss_rows, float *dl,
                              __nv_bfloat16 *dlb, cudaStream_t st);
cudaError_t launch_adam(float *w, float *m, float *v, const float *g, int64_t n, float lr, float b1, float b2, float eps,
                        float c1, float c2, const AdamTensors &T, __nv_bfloat16 *w_bf, cudaStream_t st);
cudaError_t launch_to_bf16(const float *a, int64_t n, __nv_bfloat16 *b, cudaStream_t st);

namespace {

struct Conv {
    int Cin, Cout, H, W, Ho, Wo, K, Kp;
};

constexpr int IN_H = PROPOSAL_H, IN_W = PROPOSAL_W, IN_C = 2;
constexpr int FC1_IN = 1536, FC1_OUT = 1024, FC2_OUT = PROPOSAL_CLASSES;

struct Buf {
    void *p = nullptr;
    size_t bytes = 0;
    cudaError_t ensure(size_t n)
    {
        if (n <= bytes && p) return cudaSuccess;
        if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
        cudaError_t e = cudaMalloc(&p, n < 256 ? 256 : n);
        if (e == cudaSuccess) bytes = n < 256 ? 256 : n;
        return e;
    }
    ~Buf()
    {
        if (p) cudaFree(p);
    }
    template <typename T> T *as() const { return (T *)p; }
};

// Pinned host memory, which kernels can write to as well.
struct HostBuf {
    void *p = nullptr;
    size_t bytes = 0;
    cudaError_t ensure(size_t n)
    {
        if (n <= bytes && p) return cudaSuccess;
        if (p) cudaFreeHost(p);
        p = nullptr;
        bytes = 0;
        cudaError_t e = cudaMallocHost(&p, n);
        if (e == cudaSuccess) bytes = n;
        return e;
    }
    ~HostBuf()
    {
        if (p) cudaFreeHost(p);
    }
    template <typename T> T *as() const { return (T *)p; }
};

}  // namespace

struct ProposalNet {
    Conv conv[5];
    // parameter tensors (index: conv 0..4, fc1 5, fc2 6); weights padded [N][Kp]
    int wn[7], wk[7];            // rows, padded columns
    int64_t w_off[7], b_off[7];  // offsets into the FP32 master buffers
    int64_t n_master = 0;        // total FP32 master values (padded)
    Buf master, grad, m, v, wbf; // FP32 master params/grads/Adam state; BF16 weight copies
    int64_t wbf_off[7];
    int64_t steps = 0;
    // activations (sized for the largest batch seen)
    int cap_b = 0;
    Buf col[5], y[5], h1, logits, dl, dlb, dmid, dmid_bf, dcol, part, csum;
    HostBuf status;              // written by the GEMMs only when a wait gives up
    HostBuf xfer;                // parameters or gradients on their way out
};

int64_t proposal_param_count()
{
    int64_t n = 0;
    const int cin[5] = {2, 32, 64, 64, 128}, cout[5] = {32, 64, 64, 128, 128};
    for (int l = 0; l < 5; ++l) n += (int64_t)cout[l] * 9 * cin[l] + cout[l];
    n += (int64_t)FC1_OUT * FC1_IN + FC1_OUT + (int64_t)FC2_OUT * FC1_OUT + FC2_OUT;
    return n;
}

static int pad64(int k) { return (k + 63) / 64 * 64; }

ProposalNet *proposal_create(uint64_t seed, cudaError_t *err)
{
    ProposalNet *P = new ProposalNet();
    const int cin[5] = {2, 32, 64, 64, 128}, cout[5] = {32, 64, 64, 128, 128};
    int H = IN_H, W = IN_W;
    for (int l = 0; l < 5; ++l) {
        Conv &c = P->conv[l];
        c.Cin = cin[l];
        c.Cout = cout[l];
        c.H = H;
        c.W = W;
        c.Ho = (H - 1) / 2 + 1;
        c.Wo = (W - 1) / 2 + 1;
        c.K = 9 * cin[l];
        c.Kp = pad64(c.K);
        H = c.Ho;
        W = c.Wo;
        P->wn[l] = c.Cout;
        P->wk[l] = c.Kp;
    }
    P->wn[5] = FC1_OUT;
    P->wk[5] = FC1_IN;
    P->wn[6] = FC2_OUT;
    P->wk[6] = FC1_OUT;
    int64_t o = 0, ob = 0;
    for (int t = 0; t < 7; ++t) {
        P->w_off[t] = o;
        o += (int64_t)P->wn[t] * P->wk[t];
        P->b_off[t] = o;
        o += P->wn[t];
        P->wbf_off[t] = ob;
        ob += (int64_t)P->wn[t] * P->wk[t];
    }
    P->n_master = o;
    // He-normal init (std sqrt(2 / fan_in)), zero biases; SplitMix64 + Box-Muller
    std::vector<float> h(o, 0.f);
    uint64_t state = seed;
    auto next = [&]() {
        uint64_t z = (state += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    auto uni = [&]() { return ((next() >> 11) + 0.5) * (1.0 / 9007199254740992.0); };
    for (int t = 0; t < 7; ++t) {
        const int fan_in = t < 5 ? P->conv[t].K : P->wk[t];
        const int kreal = t < 5 ? P->conv[t].K : P->wk[t];
        const double sd = std::sqrt(2.0 / fan_in);
        for (int r = 0; r < P->wn[t]; ++r)
            for (int k = 0; k < kreal; ++k) {
                const double u1 = uni(), u2 = uni();
                h[P->w_off[t] + (int64_t)r * P->wk[t] + k] =
                    (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
            }
    }
    cudaError_t e;
    if ((e = P->master.ensure(4 * o)) != cudaSuccess || (e = P->grad.ensure(4 * o)) != cudaSuccess ||
        (e = P->m.ensure(4 * o)) != cudaSuccess || (e = P->v.ensure(4 * o)) != cudaSuccess ||
        (e = P->wbf.ensure(2 * ob)) != cudaSuccess || (e = P->status.ensure(64)) != cudaSuccess) {
        *err = e;
        delete P;
        return nullptr;
    }
    cudaMemcpy(P->master.p, h.data(), 4 * o, cudaMemcpyHostToDevice);
    cudaMemset(P->grad.p, 0, 4 * o);
    cudaMemset(P->m.p, 0, 4 * o);
    cudaMemset(P->v.p, 0, 4 * o);
    memset(P->status.p, 0, 64);
    for (int t = 0; t < 7; ++t)
        launch_to_bf16(P->master.as<float>() + P->w_off[t], (int64_t)P->wn[t] * P->wk[t],
                       P->wbf.as<__nv_bfloat16>() + P->wbf_off[t], 0);
    *err = cudaDeviceSynchronize();
    if (*err != cudaSuccess) {
        delete P;
        return nullptr;
    }
    return P;
}

void proposal_destroy(ProposalNet *P) { delete P; }

// flat <-> padded master layout
static void flat_to_master(const ProposalNet *P, const float *flat, std::vector<float> &master)
{
    master.assign(P->n_master, 0.f);
    int64_t f = 0;
    for (int t = 0; t < 7; ++t) {
        const int kreal = t < 5 ? P->conv[t].K : P->wk[t];
        for (int r = 0; r < P->wn[t]; ++r)
            for (int k = 0; k < kreal; ++k) master[P->w_off[t] + (int64_t)r * P->wk[t] + k] = flat[f++];
        for (int r = 0; r < P->wn[t]; ++r) master[P->b_off[t] + r] = flat[f++];
    }
}

static void master_to_flat(const ProposalNet *P, const float *master, float *flat)
{
    int64_t f = 0;
    for (int t = 0; t < 7; ++t) {
        const int kreal = t < 5 ? P->conv[t].K : P->wk[t];
        for (int r = 0; r < P->wn[t]; ++r, f += kreal)
            memcpy(flat + f, master + P->w_off[t] + (int64_t)r * P->wk[t], sizeof(float) * kreal);
        memcpy(flat + f, master + P->b_off[t], sizeof(float) * P->wn[t]);
        f += P->wn[t];
    }
}

cudaError_t proposal_get(ProposalNet *P, int which, float *flat)
{
    cudaError_t e = P->xfer.ensure(4 * P->n_master);
    if (e != cudaSuccess) return e;
    const Buf &b = which == 0 ? P->master : P->grad;
    e = cudaMemcpy(P->xfer.p, b.p, 4 * P->n_master, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return e;
    master_to_flat(P, P->xfer.as<float>(), flat);
    return cudaSuccess;
}

cudaError_t proposal_set(ProposalNet *P, const float *flat)
{
    std::vector<float> h;
    flat_to_master(P, flat, h);
    cudaError_t e = cudaMemcpy(P->master.p, h.data(), 4 * P->n_master, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return e;
    cudaMemset(P->m.p, 0, 4 * P->n_master);
    cudaMemset(P->v.p, 0, 4 * P->n_master);
    P->steps = 0;
    for (int t = 0; t < 7; ++t)
        launch_to_bf16(P->master.as<float>() + P->w_off[t], (int64_t)P->wn[t] * P->wk[t],
                       P->wbf.as<__nv_bfloat16>() + P->wbf_off[t], 0);
    return cudaDeviceSynchronize();
}

static cudaError_t ensure_batch(ProposalNet *P, int B)
{
    if (B <= P->cap_b) return cudaSuccess;
    cudaError_t e;
    size_t max_col = 0, max_mid = 0;
    for (int l = 0; l < 5; ++l) {
        const Conv &c = P->conv[l];
        const size_t M = (size_t)B * c.Ho * c.Wo;
        if ((e = P->col[l].ensure(2 * M * c.Kp)) != cudaSuccess) return e;
        if ((e = P->y[l].ensure(2 * M * c.Cout)) != cudaSuccess) return e;
        if (l > 0) max_col = std::max(max_col, M * c.Kp);
        max_mid = std::max(max_mid, M * c.Cout);
    }
    max_mid = std::max(max_mid, (size_t)B * FC1_OUT);
    if ((e = P->h1.ensure(2 * (size_t)B * FC1_OUT)) != cudaSuccess) return e;
    if ((e = P->logits.ensure(4 * (size_t)B * FC2_OUT)) != cudaSuccess) return e;
    if ((e = P->dl.ensure(4 * (size_t)B * FC2_OUT)) != cudaSuccess) return e;
    // backward signals are carried as hi | lo BF16 pairs: twice the columns
    if ((e = P->dlb.ensure(2 * 2 * (size_t)B * FC2_OUT)) != cudaSuccess) return e;
    if ((e = P->dmid.ensure(4 * (size_t)B * FC1_IN)) != cudaSuccess) return e;      // the FC layers' input gradients
    if ((e = P->dmid_bf.ensure(2 * 2 * max_mid)) != cudaSuccess) return e;
    if ((e = P->csum.ensure(4 * (size_t)RELU_BACK_BLOCKS * FC1_IN)) != cudaSuccess) return e;
    if ((e = P->dcol.ensure(4 * max_col)) != cudaSuccess) return e;
    if ((e = P->part.ensure(4 * (size_t)32 * 1024 * 1024)) != cudaSuccess) return e;   // split-K partials
    P->cap_b = B;
    return cudaSuccess;
}

#define PK(call)                                                                                                       \
    do {                                                                                                               \
        cudaError_t e_ = (call);                                                                                       \
        if (e_ != cudaSuccess) return e_;                                                                              \
    } while (0)

// Forward pass; logits FP32 [B][64] into P->logits (and out if given).
cudaError_t proposal_forward(ProposalNet *P, const __nv_bfloat16 *in, int B, float *out, cudaStream_t st)
{
    PK(ensure_batch(P, B));
    const __nv_bfloat16 *x = in;
    const __nv_bfloat16 *wbf = P->wbf.as<__nv_bfloat16>();
    const float *mst = P->master.as<float>();
    int *status = P->status.as<int>();
    for (int l = 0; l < 5; ++l) {
        const Conv &c = P->conv[l];
        const int M = B * c.Ho * c.Wo;
        PK(launch_im2col(x, B, c.H, c.W, c.Cin, c.Ho, c.Wo, c.Kp, P->col[l].as<__nv_bfloat16>(), st));
        PK(launch_gemm_bf16(P->col[l].as<__nv_bfloat16>(), wbf + P->wbf_off[l], mst + P->b_off[l], nullptr,
                            P->y[l].as<__nv_bfloat16>(), M, c.Cout, c.Kp, c.Kp, c.Kp, c.Cout, 1, 1, nullptr, status, st));
        x = P->y[l].as<__nv_bfloat16>();
    }
    PK(launch_gemm_bf16(x, wbf + P->wbf_off[5], mst + P->b_off[5], nullptr, P->h1.as<__nv_bfloat16>(), B, FC1_OUT,
                        FC1_IN, FC1_IN, FC1_IN, FC1_OUT, 1, 1, nullptr, status, st));
    PK(launch_gemm_bf16(P->h1.as<__nv_bfloat16>(), wbf + P->wbf_off[6], mst + P->b_off[6], out ? out : P->logits.as<float>(),
                        nullptr, B, FC2_OUT, FC1_OUT, FC1_OUT, FC1_OUT, FC2_OUT, 0, 1, nullptr, status, st));
    if (out) PK(cudaMemcpyAsync(P->logits.p, out, 4 * (size_t)B * FC2_OUT, cudaMemcpyDeviceToDevice, st));
    return cudaSuccess;
}

// largest divisor of k64 = K / 64 that is <= cap
static int split_for(int K, int cap)
{
    const int k64 = K / 64;
    for (int d = std::min(cap, k64); d >= 1; --d)
        if (k64 % d == 0) return d;
    return 1;
}

// Backward signals are carried as two BF16 terms, [M][2N] = hi | lo (x ~ hi +
// lo to ~16 significant bits), so the only BF16 rounding of the backward
// pass is that of the stored forward activations and weights.

// weight gradient gW[N][Kc] = dY^T X for the split dY [M][2N] and X [M][Kc]
// (BF16), M % 64 == 0
static cudaError_t weight_grad(ProposalNet *P, const __nv_bfloat16 *dY, int M, int N, const __nv_bfloat16 *X, int Kc,
                               float *gW, cudaStream_t st)
{
    const int split = split_for(2 * M, std::max(1, (int)std::min<int64_t>(128, (int64_t)32 * 1024 * 1024 / ((int64_t)N * Kc))));
    return launch_gemm_weight_grad(dY, X, gW, M, N, Kc, split, P->part.as<float>(), P->status.as<int>(), st);
}

// One training step on a batch (B % 64 == 0): forward, loss, backward; Adam
// update if `update`.  loss_rows [B] (device or pinned host memory): the rows'
// losses.
cudaError_t proposal_train_step(ProposalNet *P, const __nv_bfloat16 *in, const int32_t *labels, int B, float lr,
                                bool update, float *loss_rows, cudaStream_t st)
{
    PK(proposal_forward(P, in, B, nullptr, st));
    float *g = P->grad.as<float>();
    __nv_bfloat16 *wbf = P->wbf.as<__nv_bfloat16>();
    PK(launch_softmax_ce(P->logits.as<float>(), labels, B, FC2_OUT, loss_rows, P->dl.as<float>(),
                         P->dlb.as<__nv_bfloat16>(), st));
    int *status = P->status.as<int>();
    float *csum = P->csum.as<float>();
    __nv_bfloat16 *dy = P->dmid_bf.as<__nv_bfloat16>();
    // FC2
    PK(weight_grad(P, P->dlb.as<__nv_bfloat16>(), B, FC2_OUT, P->h1.as<__nv_bfloat16>(), FC1_OUT, g + P->w_off[6], st));
    PK(launch_colsum(P->dlb.as<__nv_bfloat16>(), B, FC2_OUT, g + P->b_off[6], st));
    PK(launch_gemm_input_grad(P->dlb.as<__nv_bfloat16>(), wbf + P->wbf_off[6], P->dmid.as<float>(), B, FC2_OUT, FC1_OUT,
                              status, st));
    // FC1
    PK(launch_relu_back(P->dmid.as<float>(), 0, 0, 0, 0, 0, P->h1.as<__nv_bfloat16>(), B, FC1_OUT, dy, csum,
                        g + P->b_off[5], st));
    const __nv_bfloat16 *x5 = P->y[4].as<__nv_bfloat16>();
    PK(weight_grad(P, dy, B, FC1_OUT, x5, FC1_IN, g + P->w_off[5], st));
    PK(launch_gemm_input_grad(dy, wbf + P->wbf_off[5], P->dmid.as<float>(), B, FC1_OUT, FC1_IN, status, st));
    // conv layers, last to first; the gradient of layer l's output comes as dmid (l = 4: FP32, NHWC) or
    // as the dcol of layer l + 1
    for (int l = 4; l >= 0; --l) {
        const Conv &c = P->conv[l];
        const int M = B * c.Ho * c.Wo;
        if (l == 4) {
            PK(launch_relu_back(P->dmid.as<float>(), 0, 0, 0, 0, 0, P->y[l].as<__nv_bfloat16>(), M, c.Cout, dy, csum,
                                g + P->b_off[l], st));
        } else {
            const Conv &n = P->conv[l + 1];
            PK(launch_relu_back(P->dcol.as<float>(), n.H, n.W, n.Ho, n.Wo, n.Kp, P->y[l].as<__nv_bfloat16>(), M, c.Cout, dy,
                                csum, g + P->b_off[l], st));
        }
        PK(weight_grad(P, dy, M, c.Cout, P->col[l].as<__nv_bfloat16>(), c.Kp, g + P->w_off[l], st));
        if (l == 0) break;
        PK(launch_gemm_input_grad(dy, wbf + P->wbf_off[l], P->dcol.as<float>(), M, c.Cout, c.Kp, status, st));
    }
    if (update) {
        P->steps++;
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float c1 = 1.f - std::pow(b1, (float)P->steps), c2 = 1.f - std::pow(b2, (float)P->steps);
        AdamTensors T;
        for (int t = 0; t < 7; ++t) {
            T.begin[t] = P->w_off[t];
            T.end[t] = P->b_off[t];
            T.bf[t] = P->wbf_off[t];
        }
        PK(launch_adam(P->master.as<float>(), P->m.as<float>(), P->v.as<float>(), g, P->n_master, lr, b1, b2, eps, c1, c2, T,
                       wbf, st));
    }
    return cudaSuccess;
}

const float *proposal_logits(const ProposalNet *P) { return P->logits.as<float>(); }
int proposal_status(const ProposalNet *P) { return *(volatile int *)P->status.p; }

cudaError_t proposal_make_inputs(const float *const *queries, const float *renders, int n, int H, int W,
                                 __nv_bfloat16 *out, cudaStream_t st)
{
    for (int j0 = 0; j0 < n; j0 += GRAY_PAIRS) {
        const int m = std::min(GRAY_PAIRS, n - j0);
        GrayQueries q = {};
        for (int j = 0; j < m; ++j) q.img[j] = queries[j0 + j];
        PK(launch_downsample_gray(q, renders + (int64_t)j0 * 3 * H * W, m, H, W, H / IN_H,
                                  out + (int64_t)j0 * IN_H * IN_W * IN_C, st));
    }
    return cudaSuccess;
}

}  // namespace reloc
