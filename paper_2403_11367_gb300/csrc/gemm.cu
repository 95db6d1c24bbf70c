// gemm.cu -- BF16 GEMM on the 5th-generation tensor cores (tcgen05, TMEM).
//
//   C[m][n] = sum_k A[m][k] * B[n][k]   (+ bias[n], ReLU, optional)
//
// A and B are BF16; the accumulator is FP32 in tensor memory; C is written as
// FP32 or BF16.  This is the dense contraction of the learned candidate proposal
// (convolutions via im2col and the MLP, forward and backward).  An operand is
// K-major (rows of contiguous K, as above) or MN-major (stored transposed, as
// the backward pass has it: the rows of a weight gradient's operands are the
// contracted index), which the tensor cores read as it is.
//
// Persistent: as many CTAs as fit take 128 x BN output tiles (BN in {16, 32,
// ..., 256}) in turn.  A CTA of 192 threads is warp-specialised over a ring of
// shared-memory stages and two TMEM accumulators:
//   - one lane of warp 0 loads the A (128 x 64) and B (BN x 64) tiles of each
//     K step with TMA (cp.async.bulk.tensor, one box per operand: 64 BF16 =
//     128 bytes of K by the tile's rows, 128-byte swizzle, so the tiles land
//     in the canonical K-major SWIZZLE_128B layout: 128-byte rows whose 16-byte
//     chunks are XOR-permuted by the row within each 8-row, 1024-byte group)
//     and signals the stage's "full" mbarrier through the copies'
//     transaction count; the ring runs on from one tile into the next;
//   - one lane of warp 1 waits for a full stage, issues its four
//     tcgen05.mma (K = 16 each) into the tile's accumulator and commits them to
//     the stage's "empty" mbarrier, which releases the stage to the loader
//     once the MMAs have read it; after the tile's last K step it commits to the
//     accumulator's "tfull" mbarrier;
//   - warps 2..5 wait for "tfull", read the accumulator with tcgen05.ld (each
//     warp its 32 TMEM lanes), hand it back ("tempty"), and write the tile out
//     while the tensor cores work on the next one: 32 x 32 pieces go through
//     shared memory so that a row's 32 values leave as one 128-byte store (a
//     lane's own row written straight from its registers put every lane of a
//     store on another line, and the write took several times as long as the
//     tile's MMAs: a call at 8192 x 1024 x 1536 134 us, so 57 us, and 53 with the
//     waits below; 8192 x 8192 x 8192 1043 and 688).  Bias and ReLU are applied there.
// An MN-major operand's tile is loaded as boxes of 64 columns (128 bytes) by the
// 64 rows of the K step, in the canonical MN-major SWIZZLE_128B layout; its
// transposed copy (four launches per weight gradient, two per input gradient,
// 720 us of a training step of batch 256) is never made.
// With split_k > 1 a tile covers the K range [z*Ks, (z+1)*Ks) and writes FP32
// partials C[z][M][N], summed later in a fixed order.
//
// Every mbarrier wait is bounded (GEMM_WAIT_NS of the global timer): past it
// the CTA records an error in *status and every role stops at its next wait;
// the loader then waits (bounded) for its own copies in flight, the MMA lane
// commits "done" (which tracks every MMA it issued) and all threads wait for it
// (bounded) before the tensor memory is freed, so nothing the CTA started still
// writes shared or tensor memory when it exits.
#include <atomic>

#include "internal.cuh"

#include <cuda.h>

namespace reloc {

constexpr int GEMM_THREADS = 192;                   // loader, MMA, four epilogue warps
constexpr int GEMM_EPI_WARP0 = 2, GEMM_EPI_WARPS = 4;
constexpr int GEMM_BM = 128;
constexpr int GEMM_BK = 64;
constexpr int GEMM_EPI_LD = 36;                     // floats per staged row: 16-byte rows, no bank conflict
constexpr unsigned long long GEMM_WAIT_NS = 1000000000ull;   // 1 s per wait
// Tries between two looks at the timer.  A timer read before the first try and after
// every further one stood in the chain from a stage's MMAs over its refill to its
// next MMAs: 8192 x 8192 x 8192 in 128-column tiles 1360 us, 1135 so (one try that
// sleeps up to 20 us in hardware: 1178); 8192 x 1024 x 1536 57.5 -> 53.
constexpr int GEMM_TRIES = 64;
constexpr int GEMM_BAND = 16;                       // row tiles of a band of the tile order

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Shared-memory matrix descriptor of a K-major SWIZZLE_128B tile (tcgen05
// format: start >> 4 in bits 0-13, leading byte offset >> 4 in 16-29 (unused
// for swizzled K-major tiles whose K step fits the 128-byte row; 16), stride
// byte offset >> 4 in 32-45 (1024: from one 8-row group to the next), the
// fixed 0b001 in 46-48, base offset 0 (tiles start on 1024-byte
// boundaries), layout type 2 = 128-byte swizzle in 61-63).  A K step of 16
// BF16 inside the row advances the start by 32 bytes; the swizzle is applied
// to the resulting addresses.
//
// MN-major SWIZZLE_128B: 64 columns (128 bytes) of one k to a row, 8 rows to a
// 1024-byte group; the stride byte offset leads to the next 8 rows (1024), the
// leading byte offset to the next 64 columns (a box of 64 rows: 8192).  A K step
// of 16 is two groups of rows: 2048 bytes.
constexpr uint32_t MN_BOX = 64 * 64 * 2;
template <bool MN>
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((MN ? MN_BOX : 16u) >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor, kind::f16: FP32 accumulate, BF16 A and B, bits 15 and
// 16 set for an MN-major A and B, N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn ? 1u << 15 : 0u) | (b_mn ? 1u << 16 : 0u) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Wait until the phase of the given parity has completed, or GEMM_WAIT_NS.
__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(mbar), "r"(parity)
                 : "memory");
    return done != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    unsigned long long deadline = 0;
    for (;;) {
        for (int k = 0; k < GEMM_TRIES; ++k)
            if (mbar_try(mbar, parity)) return true;
        const unsigned long long now = global_ns();
        if (deadline == 0) deadline = now + GEMM_WAIT_NS;
        if (now > deadline) return false;
    }
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}

// 2D TMA load of one box at (x, y) into shared memory, completing on mbar.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t mbar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// W columns (16 or 32) of this warp's 32 TMEM lanes, one lane's row per thread.
template <int W> __device__ __forceinline__ void tmem_ld(uint32_t addr, uint32_t (&r)[W]);
template <> __device__ __forceinline__ void tmem_ld<16>(uint32_t addr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr));
}
template <> __device__ __forceinline__ void tmem_ld<32>(uint32_t addr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
                   "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
                   "=r"(r[30]), "=r"(r[31])
                 : "r"(addr));
}

struct GemmArgs {
    const float *bias;          // [N] or null
    float *Cf;                  // FP32 output (or split-K partials) or null
    __nv_bfloat16 *Cb;          // BF16 output or null
    int M, N, K;                // K multiple of 64
    int ldc;                    // row stride of C (elements)
    int relu;
    int split_k;                // >= 1; > 1 writes partials Cf[z][M][ldc]
    int n_tn, n_tiles;          // column tiles, all tiles (row tiles x column tiles x split_k)
    int vec;                    // 16-byte (BF16: 8-byte) stores allowed: ldc, N and the bases
    // MN-major operands hold half the contracted rows: K index k >= half reads
    // row k - half, of A's columns + a_xoff (the low terms of a split signal)
    int half, a_xoff;
    int inject;                 // test only: the MMA lane waits on a barrier nothing arrives at
    int *status;                // error flag (1: an mbarrier wait gave up), device or pinned host memory
};

template <int BN>
struct GemmSmem {
    static constexpr uint32_t A_BYTES = GEMM_BM * GEMM_BK * 2;
    static constexpr uint32_t B_BYTES = BN * GEMM_BK * 2;
    static constexpr uint32_t STAGE = A_BYTES + B_BYTES;
    // four stages of the widest tile fill the SM's shared memory; narrower
    // tiles need four for the loads' latency too
    static constexpr int STAGES = 4;
    static constexpr size_t EPI = (size_t)GEMM_EPI_WARPS * 32 * GEMM_EPI_LD * 4;
    static constexpr size_t TOTAL = (size_t)STAGES * STAGE + EPI + 1024;   // + alignment slack
    static constexpr uint32_t TMEM_COLS = 2 * BN < 32 ? 32 : 2 * BN;       // two accumulators, power of two >= 32
};

// Row and column tile of tile mn: bands of 16 row tiles, columns after one another
// within a band, so that the tiles in flight share their operands in both directions
// (one row of tiles after the other reads all of B again for every five rows of A).
// 8192 x 8192 x 8192: one band 714 us, bands of 16 683, of 8 700, of 32 681.
__device__ __forceinline__ int2 gemm_tile(int mn, int n_tm, int n_tn)
{
    const int per = GEMM_BAND * n_tn, band = mn / per, r = mn - band * per, rows = min(GEMM_BAND, n_tm - GEMM_BAND * band);
    return make_int2(GEMM_BAND * band + r % rows, r / rows);
}

template <int BN, bool AMN, bool BMN>
__global__ void __launch_bounds__(GEMM_THREADS)
k_gemm_bf16(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, GemmArgs g)
{
    using SM = GemmSmem<BN>;
    constexpr int STAGES = SM::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bar_full[STAGES], bar_empty[STAGES], bar_tfull[2], bar_tempty[2], bar_done,
        bar_never;
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k_per = g.K / g.split_k;                  // multiple of 64 by construction
    const int n_k = k_per / GEMM_BK;
    const int n_mn = g.n_tiles / g.split_k;
    constexpr uint32_t IDESC = instr_desc_bf16(GEMM_BM, BN, AMN, BMN);
    static_assert(!BMN || BN % 64 == 0, "whole boxes");

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)),
                     "r"(SM::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32) {
        abort_s = 0;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bar_tfull[s]), 1);
            mbar_init(smem_u32(&bar_tempty[s]), GEMM_EPI_WARPS);
        }
        mbar_init(smem_u32(&bar_done), 1);
        mbar_init(smem_u32(&bar_never), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_s;
    const uint32_t sbase = smem_u32(smem);
    // a bounded wait that gave up stops every role of the CTA
    auto wait = [&](uint64_t &bar, uint32_t parity) -> bool {
        if (mbar_try(smem_u32(&bar), parity)) return true;
        if (abort_s) return false;
        if (mbar_wait(smem_u32(&bar), parity)) return true;
        abort_s = 1;
        if (g.status) atomicExch_system(g.status, 1);
        return false;
    };

    if (tid == 0) {
        // ---- loader: the CTA's K steps, numbered through its tiles, into stage it % STAGES
        int it = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < g.n_tiles && ok; t += gridDim.x) {
            const int z = t / n_mn, mn = t - z * n_mn;
            const int2 tile = gemm_tile(mn, n_mn / g.n_tn, g.n_tn);
            const int m0 = tile.x * GEMM_BM, n0 = tile.y * BN, kbeg = z * k_per;
            for (int k = 0; k < n_k; ++k, ++it) {
                const int s = it % STAGES;
                const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
                // the stage is free once the MMAs of K step it - STAGES have read it
                if (it >= STAGES && !wait(bar_empty[s], ph ^ 1u)) { ok = false; break; }
                const uint32_t sa = sbase + s * SM::STAGE, sb = sa + SM::A_BYTES;
                const uint32_t fb = smem_u32(&bar_full[s]);
                mbar_expect_tx(fb, SM::STAGE);
                const int k0 = kbeg + k * GEMM_BK, r = k0 >= g.half ? k0 - g.half : k0;
                if (AMN) {
                    const int x = m0 + (k0 >= g.half ? g.a_xoff : 0);
                    tma_load_2d(sa, &tmA, x, r, fb);
                    tma_load_2d(sa + MN_BOX, &tmA, x + 64, r, fb);
                } else {
                    tma_load_2d(sa, &tmA, k0, m0, fb);
                }
                if (BMN) {
#pragma unroll
                    for (int j = 0; j < BN / 64; ++j) tma_load_2d(sb + j * MN_BOX, &tmB, n0 + 64 * j, r, fb);
                } else {
                    tma_load_2d(sb, &tmB, k0, n0, fb);
                }
            }
        }
        // copies still in flight land before the CTA may exit: the last one
        // issued on each stage completes that stage's current phase
        for (int i = it - STAGES < 0 ? 0 : it - STAGES; i < it; ++i)
            if (!mbar_wait(smem_u32(&bar_full[i % STAGES]), (uint32_t)(i / STAGES) & 1u) && g.status)
                atomicExch_system(g.status, 1);
    } else if (tid == 32) {
        // ---- MMA issuer ----------------------------------------------------------
        bool ok = true;
        if (g.inject) ok = wait(bar_never, 0u);          // test only: a wait that nothing completes runs out
        int it = 0, i = 0;
        for (int t = blockIdx.x; t < g.n_tiles && ok; t += gridDim.x, ++i) {
            // the accumulator is free once the epilogue of tile i - 2 has read it
            if (i >= 2 && !wait(bar_tempty[i & 1], ((uint32_t)(i >> 1) & 1u) ^ 1u)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t acc_t = tmem + (uint32_t)((i & 1) * BN);
            for (int k = 0; k < n_k; ++k, ++it) {
                const int s = it % STAGES;
                if (!wait(bar_full[s], (uint32_t)(it / STAGES) & 1u)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t sa = sbase + s * SM::STAGE, sb = sa + SM::A_BYTES;
#pragma unroll
                for (int j = 0; j < GEMM_BK / 16; ++j) {
                    // K step j: 16 BF16 = 32 bytes further along the 128-byte rows, or 16 rows on
                    const uint64_t da = smem_desc_sw128<AMN>(sa + (AMN ? 2048 : 32) * j);
                    const uint64_t db = smem_desc_sw128<BMN>(sb + (BMN ? 2048 : 32) * j);
                    const uint32_t acc = (k > 0 || j > 0) ? 1u : 0u;
                    asm volatile("{\n\t.reg .pred p;\n\t"
                                 "setp.ne.u32 p, %4, 0;\n\t"
                                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(acc_t),
                                 "l"(da), "l"(db), "r"(IDESC), "r"(acc)
                                 : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(smem_u32(&bar_empty[s]))
                             : "memory");
            }
            if (ok)
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(smem_u32(&bar_tfull[i & 1]))
                             : "memory");
        }
        // "done" completes once every MMA this lane issued has finished
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     ::"r"(smem_u32(&bar_done))
                     : "memory");
    } else if (warp >= GEMM_EPI_WARP0) {
        // ---- epilogue: TMEM -> registers -> shared memory -> global -----------------
        constexpr int CW = BN < 32 ? BN : 32;           // columns per piece
        const int quad = warp & 3;                      // the 32 TMEM lanes this warp may read
        float *const st = reinterpret_cast<float *>(smem + (size_t)STAGES * SM::STAGE) +
                          (warp - GEMM_EPI_WARP0) * 32 * GEMM_EPI_LD;
        int i = 0;
        for (int t = blockIdx.x; t < g.n_tiles; t += gridDim.x, ++i) {
            const int z = t / n_mn, mn = t - z * n_mn;
            const int2 tile = gemm_tile(mn, n_mn / g.n_tn, g.n_tn);
            const int row0 = tile.x * GEMM_BM + quad * 32, n0 = tile.y * BN;
            // every lane waits for itself; one that gave up takes the warp out
            if (!__all_sync(0xffffffffu, wait(bar_tfull[i & 1], (uint32_t)(i >> 1) & 1u))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t src = tmem + (uint32_t)((i & 1) * BN) + ((uint32_t)(quad * 32) << 16);
            const int rows = min(32, g.M - row0);
            const int64_t crow = (int64_t)z * g.M * (g.split_k > 1) + row0;
#pragma unroll 1
            for (int c0 = 0; c0 < BN; c0 += CW) {
                uint32_t r[CW];
                tmem_ld<CW>(src + c0, r);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (c0 + CW == BN) {
                    // the accumulator is read: hand it back before the last stores
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bar_tempty[i & 1]));
                }
                if (n0 + c0 >= g.N || rows <= 0) continue;   // uniform over the warp
                __syncwarp();
#pragma unroll
                for (int c = 0; c < CW; c += 4)
                    *reinterpret_cast<float4 *>(st + lane * GEMM_EPI_LD + c) =
                        make_float4(__uint_as_float(r[c]), __uint_as_float(r[c + 1]), __uint_as_float(r[c + 2]),
                                    __uint_as_float(r[c + 3]));
                __syncwarp();
                const int cn = min(CW, g.N - n0 - c0);      // valid columns of the piece
                if (g.vec) {
                    constexpr int LPR = CW / 4, RPS = 32 / LPR;   // lanes per row, rows per store
                    const int c = (lane % LPR) * 4, col = n0 + c0 + c;
                    if (c < cn) {                           // N is a multiple of 4: whole groups
                        float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (g.bias) b = make_float4(g.bias[col], g.bias[col + 1], g.bias[col + 2], g.bias[col + 3]);
#pragma unroll
                        for (int rr = lane / LPR; rr < 32; rr += RPS) {
                            if (rr >= rows) break;
                            float4 v = *reinterpret_cast<const float4 *>(st + rr * GEMM_EPI_LD + c);
                            if (g.bias) { v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w; }
                            if (g.relu) {
                                v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f);
                                v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f);
                            }
                            const int64_t o = (crow + rr) * g.ldc + col;
                            if (g.Cf) *reinterpret_cast<float4 *>(g.Cf + o) = v;
                            if (g.Cb) {
                                __nv_bfloat162 h[2] = {__floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(v.z, v.w)};
                                *reinterpret_cast<uint2 *>(g.Cb + o) = *reinterpret_cast<const uint2 *>(h);
                            }
                        }
                    }
                } else if (lane < cn) {
                    const int col = n0 + c0 + lane;
                    const float b = g.bias ? g.bias[col] : 0.f;
                    for (int rr = 0; rr < rows; ++rr) {
                        float v = st[rr * GEMM_EPI_LD + lane];
                        if (g.bias) v += b;
                        if (g.relu) v = fmaxf(v, 0.f);
                        const int64_t o = (crow + rr) * g.ldc + col;
                        if (g.Cf) g.Cf[o] = v;
                        if (g.Cb) g.Cb[o] = __float2bfloat16_rn(v);
                    }
                }
            }
        }
    }
    __syncwarp();
    __syncthreads();
    if (!mbar_wait(smem_u32(&bar_done), 0u) && g.status) atomicExch_system(g.status, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SM::TMEM_COLS) : "memory");
}

// Sum split-K partials in a fixed order and apply the epilogue.
__global__ void k_gemm_reduce(const float *__restrict__ part, int split, int M, int N, int ldc,
                              const float *__restrict__ bias, int relu, float *__restrict__ Cf,
                              __nv_bfloat16 *__restrict__ Cb)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)M * N) return;
    const int row = (int)(i / N), col = (int)(i % N);
    // eight partials in flight, added in order (few outputs of many partials
    // leave the loop waiting for one load at a time otherwise)
    float v = 0.f;
    const float *p = part + (int64_t)row * ldc + col;
    const int64_t step = (int64_t)M * ldc;
    int z = 0;
    for (; z + 8 <= split; z += 8) {
        float x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = p[(z + j) * step];
#pragma unroll
        for (int j = 0; j < 8; ++j) v += x[j];
    }
    for (; z < split; ++z) v += p[z * step];
    if (bias) v += bias[col];
    if (relu) v = fmaxf(v, 0.f);
    if (Cf) Cf[(int64_t)row * ldc + col] = v;
    if (Cb) Cb[(int64_t)row * ldc + col] = __float2bfloat16_rn(v);
}

// ---- tensor maps ---------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled()
{
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
        else
            cudaGetLastError();
    }
    return fn;
}

// Row-major BF16 matrix [rows][ld], cols used, in boxes of 64 columns (128 bytes)
// by box_rows rows, 128-byte swizzle; what lies beyond rows or cols reads 0.
static cudaError_t make_map(CUtensorMap *map, const __nv_bfloat16 *base, int rows, int cols, int ld, int box_rows)
{
    EncodeTiledFn fn = encode_tiled();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t stride[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)base, dim, stride, box, estride,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// An operand as it lies in memory: rows x cols used of row stride ld.
struct GemmOperand {
    const __nv_bfloat16 *p;
    int rows, cols, ld;
};

// CTAs of k_gemm_bf16 that fit on the current device at once: by shared
// memory and registers, and at most 512 TMEM columns to an SM.  0 on error.
template <int BN, bool AMN, bool BMN>
static int gemm_resident()
{
    constexpr int MAX_DEV = 64;
    static std::atomic<int> cached[MAX_DEV];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return 0;
    int c = cached[dev].load();
    if (!c) {
        int sms = 0, per_sm = 0;
        if (cudaFuncSetAttribute(k_gemm_bf16<BN, AMN, BMN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)GemmSmem<BN>::TOTAL) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemm_bf16<BN, AMN, BMN>, GEMM_THREADS,
                                                          GemmSmem<BN>::TOTAL) != cudaSuccess)
            return 0;
        const int by_tmem = 512 / (int)GemmSmem<BN>::TMEM_COLS;
        c = sms * (per_sm < 1 ? 1 : per_sm < by_tmem ? per_sm : by_tmem);
        cached[dev].store(c);
    }
    return c;
}

template <int BN, bool AMN, bool BMN>
static cudaError_t gemm_t(const GemmOperand &A, const GemmOperand &B, GemmArgs g, cudaStream_t st)
{
    CUtensorMap ma, mb;
    cudaError_t e = make_map(&ma, A.p, A.rows, A.cols, A.ld, AMN ? GEMM_BK : GEMM_BM);
    if (e == cudaSuccess) e = make_map(&mb, B.p, B.rows, B.cols, B.ld, BMN ? GEMM_BK : BN);
    if (e != cudaSuccess) return e;
    const int resident = gemm_resident<BN, AMN, BMN>();
    if (resident <= 0) {
        e = cudaGetLastError();
        return e != cudaSuccess ? e : cudaErrorInvalidValue;
    }
    g.n_tn = (int)ceil_div(g.N, BN);
    const int64_t tiles = ceil_div(g.M, GEMM_BM) * g.n_tn * g.split_k;
    if (tiles > (int64_t)1 << 30) return cudaErrorInvalidValue;
    g.n_tiles = (int)tiles;
    k_gemm_bf16<BN, AMN, BMN><<<(unsigned)min64(tiles, resident), GEMM_THREADS, GemmSmem<BN>::TOTAL, st>>>(ma, mb, g);
    return cudaGetLastError();
}

// The widest tile that N fills, halved while that shortens the busiest SM's time: its
// rounds of one tile times a K step's, which goes with BN + 600 (8192 x 8192 x 8192: 0.383
// us a step at 256 columns, 0.326 at 128, 0.297 at 64, 0.292 at 32; the chain from a
// stage's MMAs over its refill does not shorten with the tile).  So narrow tiles pay only
// where they cost no round: 128 rows by 1024 columns would run on 4 SMs at BN = 256.
// Counting the columns of a round alone took 128 for that product, 1074 us, so 688; 32
// for 5000 x 2000 x 1024, 94 us, so 31.
constexpr int GEMM_STEP_COLUMNS = 600;
static int gemm_bn(int M, int N, int split_k, int least)
{
    int BN = N <= 16 ? 16 : N <= 32 ? 32 : N <= 64 ? 64 : N <= 128 ? 128 : 256;
    if (BN < least) BN = least;
    auto time = [&](int bn) {
        return ceil_div(ceil_div(M, GEMM_BM) * ceil_div(N, bn) * split_k, 152) * (bn + GEMM_STEP_COLUMNS);
    };
    while (BN / 2 >= (least > 32 ? least : 32) && time(BN / 2) < time(BN)) BN /= 2;
    return BN;
}

// Fills in the output side of g and runs the epilogue's reduction after `run`.
template <typename F>
static cudaError_t gemm_split(GemmArgs &g, const float *bias, float *Cf, __nv_bfloat16 *Cb, int M, int N, int K, int ldc,
                              int relu, int split_k, float *partials, int *status, cudaStream_t st, int inject, F run)
{
    g.bias = bias; g.Cf = Cf; g.Cb = Cb;
    g.M = M; g.N = N; g.K = K; g.ldc = ldc;
    g.relu = relu; g.split_k = split_k; g.status = status;
    g.inject = take_fault(FAULT_GEMM_WAIT) ? 1 : inject;
    if (split_k > 1) {
        g.Cf = partials;
        g.Cb = nullptr;
        g.bias = nullptr;
        g.relu = 0;
    }
    g.vec = N % 4 == 0 && ldc % 4 == 0 && ((uintptr_t)g.Cf & 15) == 0 && ((uintptr_t)g.Cb & 7) == 0;
    cudaError_t e = run();
    if (e != cudaSuccess || split_k == 1) return e;
    const int64_t n = (int64_t)M * N;
    k_gemm_reduce<<<(unsigned)ceil_div(n, 256), 256, 0, st>>>(partials, split_k, M, N, ldc, bias, relu, Cf, Cb);
    return cudaGetLastError();
}

// C = A B^T (+ bias, ReLU).  Requirements: K % 64 == 0, K / split_k % 64 == 0,
// lda, ldb multiples of 8 (16-byte rows), 16-byte aligned A and B.
// split_k > 1 needs `partials` (split_k * M * ldc floats).  inject != 0, or a
// pending FAULT_GEMM_WAIT injection (tests only), makes the CTAs' MMA lanes
// wait on a barrier nothing completes: every CTA gives up after the wait
// limit, issues no MMA and sets *status.
cudaError_t launch_gemm_bf16(const __nv_bfloat16 *A, const __nv_bfloat16 *B, const float *bias, float *Cf,
                             __nv_bfloat16 *Cb, int M, int N, int K, int lda, int ldb, int ldc, int relu, int split_k,
                             float *partials, int *status, cudaStream_t st, int inject)
{
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    if (K % GEMM_BK || split_k < 1 || (K / split_k) % GEMM_BK || (lda % 8) || (ldb % 8) ||
        ((uintptr_t)A & 15) || ((uintptr_t)B & 15) || (split_k > 1 && !partials))
        return cudaErrorInvalidValue;
    GemmArgs g{};
    g.half = K;                                          // no second half
    const GemmOperand a{A, M, K, lda}, b{B, N, K, ldb};
    return gemm_split(g, bias, Cf, Cb, M, N, K, ldc, relu, split_k, partials, status, st, inject, [&]() {
        switch (gemm_bn(M, N, split_k, 16)) {
        case 16: return gemm_t<16, false, false>(a, b, g, st);
        case 32: return gemm_t<32, false, false>(a, b, g, st);
        case 64: return gemm_t<64, false, false>(a, b, g, st);
        case 128: return gemm_t<128, false, false>(a, b, g, st);
        default: return gemm_t<256, false, false>(a, b, g, st);
        }
    });
}

// Weight gradient gW [N][Kc] = (hi + lo)^T X for a split signal dY [R][2 N] (hi |
// lo) and X [R][Kc]: the contraction runs over the 2 R rows hi then lo, X read
// twice, both operands as they lie.  R a multiple of 64, N and Kc of 8.
cudaError_t launch_gemm_weight_grad(const __nv_bfloat16 *dY, const __nv_bfloat16 *X, float *gW, int R, int N, int Kc,
                                    int split_k, float *partials, int *status, cudaStream_t st)
{
    const int K = 2 * R;
    if (R <= 0 || R % GEMM_BK || N % 8 || Kc % 8 || split_k < 1 || (K / GEMM_BK) % split_k ||
        ((uintptr_t)dY & 15) || ((uintptr_t)X & 15) || (split_k > 1 && !partials))
        return cudaErrorInvalidValue;
    GemmArgs g{};
    g.half = R;
    g.a_xoff = N;
    const GemmOperand a{dY, R, 2 * N, 2 * N}, b{X, R, Kc, Kc};
    return gemm_split(g, nullptr, gW, nullptr, N, Kc, K, Kc, 0, split_k, partials, status, st, 0, [&]() {
        switch (gemm_bn(N, Kc, split_k, 64)) {
        case 64: return gemm_t<64, true, true>(a, b, g, st);
        case 128: return gemm_t<128, true, true>(a, b, g, st);
        default: return gemm_t<256, true, true>(a, b, g, st);
        }
    });
}

// Input gradient dX [R][Kc] = (hi + lo) W for a split signal dY [R][2 N] and the
// weights W [N][Kc] as they lie (read twice).  N a multiple of 64, Kc of 8.
cudaError_t launch_gemm_input_grad(const __nv_bfloat16 *dY, const __nv_bfloat16 *W, float *dX, int R, int N, int Kc,
                                   int *status, cudaStream_t st)
{
    if (R <= 0 || N % GEMM_BK || Kc % 8 || ((uintptr_t)dY & 15) || ((uintptr_t)W & 15)) return cudaErrorInvalidValue;
    GemmArgs g{};
    g.half = N;
    const GemmOperand a{dY, R, 2 * N, 2 * N}, b{W, N, Kc, Kc};
    return gemm_split(g, nullptr, dX, nullptr, R, Kc, 2 * N, Kc, 0, 1, nullptr, status, st, 0, [&]() {
        switch (gemm_bn(R, Kc, 1, 64)) {
        case 64: return gemm_t<64, false, true>(a, b, g, st);
        case 128: return gemm_t<128, false, true>(a, b, g, st);
        default: return gemm_t<256, false, true>(a, b, g, st);
        }
    });
}

}  // namespace reloc
