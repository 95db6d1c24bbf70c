// sort.cu -- depth ordering and tile binning of the projected Gaussians.
//
// Sec. III-A of 3DGS-ReLoc composites each pixel's Gaussians "sorted by
// depth".  Per view the required order of a tile's list is (depth, Gaussian
// index).  It is produced without any sort over the (much larger) instance
// list:
//   1. a stable LSD radix sort of the visible (view, Gaussian) pairs by the
//      float32 depth bit pattern (4 passes of 8 bits; the first pass also
//      drops invisible pairs, so compaction costs nothing extra): one
//      thread-block cluster per view runs all four passes (k_depth_sort), and
//      views of more Gaussians than that suits take a launch chain per pass;
//   2. per chunk of that depth order, tile coverage counts (K3: 2D difference
//      arrays), scanned into each tile's list start and each chunk's slot in it;
//   3. emission of every (tile, Gaussian) instance straight into its slot, a
//      warp per (chunk, tile row) walking the chunk in depth order (K4).
// Stability of the depth sort makes every tile's list ordered by depth and,
// for equal depth bits, by Gaussian index -- the same order as one stable sort
// of view|tile|depth keys emitted in index order.
//
// Every per-view array sits at a host-planned offset with a host-planned
// capacity, and chunk tables map a block to its view and chunk, so valid
// lengths stay in device memory: no host round trip between stages.
#include <atomic>

#include <cooperative_groups.h>

#include "internal.cuh"

namespace reloc {

static_assert(SORT_THREADS == RADIX, "scatter assigns one digit per thread");

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Block-wide exclusive scan of one value per thread; *total gets the sum.
// s_tmp: 33 words of shared memory.  All threads must call it.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t *s_tmp, uint32_t *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_tmp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nw ? s_tmp[lane] : 0u, wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        s_tmp[lane] = wi - w;
        if (lane == 31) s_tmp[32] = wi;
    }
    __syncthreads();
    uint32_t r = s_tmp[warp] + inc - x;
    *total = s_tmp[32];
    __syncthreads();
    return r;
}

// --------------------------------------------- depth sort, one launch ------
// A cluster of C blocks (1 .. 16, a power of two) per view runs the four passes
// of the stable LSD sort.  Per pass, block r takes the r-th share of the items
// and warp w the w-th share of those:
//   count    each warp counts its items' digits in its own shared-memory
//            histogram;
//   offsets  the blocks' digit counts are read across the cluster (distributed
//            shared memory), and digit d of warp w of block r starts at the
//            total of the smaller digits, plus digit d of the blocks before r,
//            plus digit d of the warps before w;
//   scatter  each warp walks its items again in order, 32 at a time, ranks the
//            lanes of equal digit by ballots and writes (key, index) straight
//            to its place.
// Cluster barriers (release / acquire, so they order the items in global memory
// too) stand between the passes.  Pass 0 reads the view's dense depth keys and
// drops the culled ones, the last pass writes indices only.
// What bounds it: for few views the latency of the four dependent passes (12
// launches of 4 to 7 us each as a chain: 76 us for one driving view of 320k keys,
// 104k of them visible, 50 us so; 72 and 27 us for one of 10k), for many the
// scattered 8-byte stores, about one lane a clock and SM (64 driving views 470 us
// as a chain, 278 us so).  The first items of each lane stay in registers
// between count and scatter; the cluster's counts are read with all loads in
// flight (one after the other they cost more than the pass's items: 88 us for the
// one driving view).  Shared memory holds counters only, so a view's visible count
// is not bounded by it.
constexpr int DS_MAX_CLUSTER = 16;
constexpr int DS_WIDE_VIEWS = 8;
constexpr int DS_KEPT0 = 16, DS_KEPT = 8;            // items per lane kept in registers between count and scatter
constexpr int DS_UNROLL = 4;                         // further items per lane in flight

template <int NW>
struct DepthSortShared {
    uint32_t w[NW][RADIX];                           // a warp's digit counts, then its running offsets
    uint32_t cnt[RADIX];                             // the block's digit counts, read by the whole cluster
    uint32_t tmp[33];
};

// One pass over n items: of dense keys (FIRST: culled ones dropped, values the
// positions) or (key, value) pairs, to pairs or (LAST) values.  Returns the
// items kept.
template <int NW, bool FIRST, bool LAST>
__device__ __forceinline__ uint32_t depth_sort_pass(DepthSortShared<NW> &sm, uint32_t n, int shift,
                                                    const uint32_t *__restrict__ keys, const uint2 *src, uint2 *dst,
                                                    uint32_t *out)
{
    namespace cg = cooperative_groups;
    constexpr int KEPT = FIRST ? DS_KEPT0 : DS_KEPT;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = lanemask_lt();
    uint32_t *const sw = sm.w[warp];
    // this block's and this warp's shares, whole rounds of 32
    const uint32_t per_b = ((n + C - 1) / C + 31) / 32 * 32;
    const uint32_t b0 = min(n, rank * per_b), b1 = min(n, b0 + per_b);
    const uint32_t per_w = ((b1 - b0 + NW - 1) / NW + 31) / 32 * 32;
    const uint32_t w0 = min(b1, b0 + warp * per_w), w1 = min(b1, w0 + per_w);
    auto load = [&](uint32_t i, uint2 &t) {
        if (i < w1) {
            if (FIRST) t.x = __ldg(keys + i);
            else t = src[i];
        }
    };
    // digit of item i (RADIX: none)
    auto digit = [&](uint32_t i, const uint2 &t) -> uint32_t {
        if (i >= w1 || (FIRST && t.x == 0xFFFFFFFFu)) return (uint32_t)RADIX;
        return (t.x >> shift) & 255u;
    };
    uint2 kept[KEPT];
#pragma unroll
    for (int u = 0; u < KEPT; ++u) load(w0 + lane + 32 * u, kept[u]);
    for (int d = lane; d < RADIX; d += 32) sw[d] = 0;
    __syncwarp();
#pragma unroll
    for (int u = 0; u < KEPT; ++u) {
        const uint32_t d = digit(w0 + lane + 32 * u, kept[u]);
        if (d != (uint32_t)RADIX) atomicAdd(sw + d, 1u);
    }
    for (uint32_t i = w0 + lane + 32 * KEPT; i < w1; i += 32 * DS_UNROLL) {
        uint2 t[DS_UNROLL];
#pragma unroll
        for (int u = 0; u < DS_UNROLL; ++u) load(i + 32 * u, t[u]);
#pragma unroll
        for (int u = 0; u < DS_UNROLL; ++u) {
            const uint32_t d = digit(i + 32 * u, t[u]);
            if (d != (uint32_t)RADIX) atomicAdd(sw + d, 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x < RADIX) {
        uint32_t c = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) c += sm.w[w][threadIdx.x];
        sm.cnt[threadIdx.x] = c;
    }
    cl.sync();
    uint32_t total = 0, before = 0;
    if (threadIdx.x < RADIX) {
        uint32_t c[DS_MAX_CLUSTER];                  // all the remote loads in flight
#pragma unroll
        for (int r = 0; r < DS_MAX_CLUSTER; ++r) c[r] = r < C ? cl.map_shared_rank(sm.cnt, r)[threadIdx.x] : 0u;
#pragma unroll
        for (int r = 0; r < DS_MAX_CLUSTER; ++r) {
            before += r < rank ? c[r] : 0u;
            total += c[r];
        }
    }
    uint32_t all;
    uint32_t run = block_excl_scan(total, sm.tmp, &all) + before;
    if (threadIdx.x < RADIX) {
        uint32_t c[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) c[w] = sm.w[w][threadIdx.x];
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            sm.w[w][threadIdx.x] = run;
            run += c[w];
        }
    }
    __syncthreads();
    auto place = [&](uint32_t i, const uint2 &t) {
        const uint32_t d = digit(i, t);
        // lanes holding the same digit (or none): the intersection of nine
        // ballots, one per bit of d (0 .. RADIX)
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < 9; ++b) {
            const bool set = ((d >> b) & 1u) != 0u;
            const unsigned bal = __ballot_sync(0xffffffffu, set);
            peers &= set ? bal : ~bal;
        }
        const bool valid = d != (uint32_t)RADIX;
        uint32_t at = 0;
        if (valid) at = sw[d];
        __syncwarp();
        if (valid && (peers & lt) == 0) sw[d] = at + __popc(peers);
        __syncwarp();
        if (valid) {
            at += __popc(peers & lt);
            if (LAST) out[at] = t.y;
            else dst[at] = FIRST ? make_uint2(t.x, i) : t;
        }
    };
#pragma unroll
    for (int u = 0; u < KEPT; ++u)
        if (w0 + 32 * u < w1) place(w0 + lane + 32 * u, kept[u]);        // uniform over the warp
    for (uint32_t i = w0 + 32 * KEPT; i < w1; i += 32 * DS_UNROLL) {
        uint2 t[DS_UNROLL];
#pragma unroll
        for (int u = 0; u < DS_UNROLL; ++u) load(i + lane + 32 * u, t[u]);
#pragma unroll
        for (int u = 0; u < DS_UNROLL; ++u)
            if (i + 32 * u < w1) place(i + lane + 32 * u, t[u]);
    }
    cl.sync();                                       // items written; the counts may be rewritten (and the block may exit)
    return all;
}

template <int NW>
__global__ void __launch_bounds__(32 * NW, NW == 16 ? 2 : 1)
k_depth_sort(const uint32_t *__restrict__ dkey, uint2 *bufA, uint2 *bufB, uint32_t *out, Layout L, uint32_t *n_vis)
{
    __shared__ DepthSortShared<NW> sm;
    chain_wait();
    const int C = (int)cooperative_groups::this_cluster().num_blocks();
    const int v = blockIdx.x / C;
    const int64_t off = L.vd_off[v];
    uint2 *const A = bufA + off, *const B = bufB + off;
    uint32_t n = (uint32_t)(L.vd_off[v + 1] - off);
    n = depth_sort_pass<NW, true, false>(sm, n, 0, dkey + off, nullptr, A, nullptr);
    if (blockIdx.x % C == 0 && threadIdx.x == 0) n_vis[v] = n;
    depth_sort_pass<NW, false, false>(sm, n, 8, nullptr, A, B, nullptr);
    depth_sort_pass<NW, false, false>(sm, n, 16, nullptr, B, A, nullptr);
    depth_sort_pass<NW, false, true>(sm, n, 24, nullptr, A, nullptr, out + off);
}

// Blocks of the largest cluster of k_depth_sort<NW> that the current device can place
// (16 is beyond the portable 8; a device with fewer usable SMs in its GPCs takes less), 0
// on error; asked once per device.
template <int NW>
static int depth_sort_cluster()
{
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int c = cached[dev].load();
    for (int C = DS_MAX_CLUSTER; !c && C >= 1; C /= 2) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = C;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(32 * NW);
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_depth_sort<NW>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        if (n > 0) cached[dev].store(c = C);
    }
    return c;
}

cudaError_t launch_depth_sort(const uint32_t *dkey, uint2 *bufA, uint2 *bufB, uint32_t *out, const Layout &L,
                              int64_t longest, uint32_t *n_vis, cudaStream_t st)
{
    if (L.V <= 0) return cudaSuccess;
    // one block per 2048 keys of the longest view, at most the whole cluster, and
    // half of it once the views alone fill the GPU: 64 driving views 278 us at 8
    // blocks, 339 at 16, 298 at 4; 16 views 153 at 16, 168 at 8; one view 50 at
    // 16, 77 at 8; a view of 10k keys 27 at 8, 35 at 2
    const bool wide = L.V <= DS_WIDE_VIEWS;
    const int fits = wide ? depth_sort_cluster<32>() : depth_sort_cluster<16>();
    if (fits <= 0) return cudaErrorInvalidConfiguration;
    const int most = min(fits, L.V <= 32 ? DS_MAX_CLUSTER : DS_MAX_CLUSTER / 2);
    int C = 1;
    while (C < most && (int64_t)C * 2048 < longest) C *= 2;
    const dim3 grid((unsigned)(C * L.V));
    return wide ? launch_chained(k_depth_sort<32>, grid, dim3(1024), 0, st, C, dkey, bufA, bufB, out, L, n_vis)
                : launch_chained(k_depth_sort<16>, grid, dim3(512), 0, st, C, dkey, bufA, bufB, out, L, n_vis);
}

// --------------------------------------- depth sort, launches per pass -----
// For views of more Gaussians than a cluster suits (DEPTH_SORT_CLUSTER_VISIBLE),
// whose passes need the whole GPU: upsweep, digit offsets and scatter over SORT_CHUNK items a
// block.
// Per chunk digit counts -> hist[s][d][k] (digit-major inside a segment, so
// one exclusive scan of the segment's block gives every chunk's offsets).
// Each key adds 1 to its warp's own histogram with a shared-memory atomic;
// the warps' histograms are summed at the end.  (Merging a warp's equal
// digits first with __match_any_sync, one atomic per distinct digit, kept
// the MIO queue full: the depth sort took 0.66 instead of 0.51 ms per
// 64-candidate query, on the exponent byte too, where few values recur.)
__global__ void __launch_bounds__(SORT_THREADS) k_radix_upsweep(RadixPass p)
{
    constexpr int NW = SORT_THREADS / 32;
    __shared__ uint32_t s_h[NW][RADIX];
    const int c = blockIdx.x;
    const int s = find_segment(p.chunk_base, p.n_seg, c);
    const int k = c - p.chunk_base[s], cps = p.chunk_base[s + 1] - p.chunk_base[s];
    const int warp = threadIdx.x >> 5;
#pragma unroll
    for (int w = 0; w < NW; ++w) s_h[w][threadIdx.x] = 0;
    __syncthreads();
    const int64_t cap = p.seg_off[s + 1] - p.seg_off[s];
    const int64_t seg_len = p.len ? min64(p.len[s], cap) : cap;
    const int64_t begin = (int64_t)k * SORT_CHUNK;
    const int n = (int)max64(0, min64(SORT_CHUNK, seg_len - begin));
    const int64_t base = p.seg_off[s] + begin;
    // all of this thread's loads first (independent, in flight together), then the counts
    uint32_t d[SORT_IPT];
#pragma unroll
    for (int r = 0; r < SORT_IPT; ++r) {
        const int idx = r * SORT_THREADS + threadIdx.x;
        d[r] = RADIX;
        if (idx < n) {
            const uint32_t k = p.keys_in[base + idx];
            const bool keep = !p.drop_culled || k != 0xFFFFFFFFu;
            d[r] = keep ? (k >> p.shift) & p.mask : (uint32_t)RADIX;
        }
    }
#pragma unroll
    for (int r = 0; r < SORT_IPT; ++r)
        if (d[r] != (uint32_t)RADIX) atomicAdd(&s_h[warp][d[r]], 1u);
    __syncthreads();
    uint32_t cnt = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) cnt += s_h[w][threadIdx.x];
    p.hist[(int64_t)RADIX * p.chunk_base[s] + (int64_t)threadIdx.x * cps + k] = cnt;
    if (cnt) atomicAdd(p.dtot + (int64_t)RADIX * s + threadIdx.x, cnt);
}

// ------------------------------------------------------- digit offsets -----
// Exclusive offsets of one pass in place: the segment's counts are stored
// digit-major ([digit][chunk]), so the offset of (d, k) is the total of all
// smaller digits (dtot, summed by the upsweep) plus the counts of digit d in
// the chunks before k.  A warp per (segment, digit) takes the first from
// dtot and scans the second 32 chunks at a time; len_out[s] (may be null) =
// the segment's total.
constexpr int DSCAN_WARPS = 8;
__global__ void __launch_bounds__(32 * DSCAN_WARPS)
k_digit_scan(uint32_t *hist, const uint32_t *__restrict__ dtot, const int32_t *__restrict__ chunk_base,
             uint32_t *len_out)
{
    const int s = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int d = blockIdx.y * DSCAN_WARPS + warp;
    const uint32_t *dt = dtot + (int64_t)RADIX * s;
    uint32_t below = 0, all = 0;
    for (int i = lane; i < RADIX; i += 32) {
        const uint32_t x = dt[i];
        below += i < d ? x : 0u;
        all += x;
    }
    below = __reduce_add_sync(0xffffffffu, below);
    all = __reduce_add_sync(0xffffffffu, all);
    if (len_out && d == 0 && lane == 0) len_out[s] = all;
    const int cps = chunk_base[s + 1] - chunk_base[s];
    uint32_t *h = hist + (int64_t)RADIX * chunk_base[s] + (int64_t)d * cps;
    uint32_t carry = below;
    for (int k0 = 0; k0 < cps; k0 += 32) {
        const int k = k0 + lane;
        const uint32_t x = k < cps ? h[k] : 0u;
        uint32_t inc = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (k < cps) h[k] = carry + inc - x;
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
}

// ------------------------------------------------------------ scatter ------
// Stable scatter of one chunk.  Warp w owns the contiguous items
// [w*256, (w+1)*256) and ranks them round by round (the lanes sharing a
// digit from nine ballots, one per bit of the digit), so ranks follow input
// order; per-warp digit counters then give each warp's offset inside the
// block.  Items are staged digit-sorted in shared memory and written out in
// runs (coalesced).
__global__ void __launch_bounds__(SORT_THREADS) k_radix_scatter(RadixPass p)
{
    constexpr int NW = SORT_THREADS / 32;
    __shared__ uint32_t s_wcnt[NW][RADIX];
    __shared__ uint32_t s_boff[RADIX];
    __shared__ uint32_t s_goff[RADIX];
    __shared__ uint32_t s_key[SORT_CHUNK];
    __shared__ uint32_t s_val[SORT_CHUNK];
    __shared__ uint32_t s_tmp[33];

    const int c = blockIdx.x;
    const int s = find_segment(p.chunk_base, p.n_seg, c);
    const int k = c - p.chunk_base[s], cps = p.chunk_base[s + 1] - p.chunk_base[s];
    const int64_t cap = p.seg_off[s + 1] - p.seg_off[s];
    const int64_t seg_len = p.len ? min64(p.len[s], cap) : cap;
    const int64_t begin = (int64_t)k * SORT_CHUNK;
    if (begin >= seg_len) return;                       // uniform for the block
    const int n = (int)min64(SORT_CHUNK, seg_len - begin);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int w = 0; w < NW; ++w) s_wcnt[w][threadIdx.x] = 0;
    __syncthreads();

    const int64_t base = p.seg_off[s] + begin;
    const unsigned lt = lanemask_lt();
    uint32_t key[SORT_IPT], val[SORT_IPT], rank[SORT_IPT];
    bool vld[SORT_IPT];
    // all of this thread's loads first (independent, in flight together), then the ranks
#pragma unroll
    for (int r = 0; r < SORT_IPT; ++r) {
        const int idx = warp * (32 * SORT_IPT) + r * 32 + lane;
        vld[r] = idx < n;
        key[r] = 0u;
        val[r] = 0u;
        if (vld[r]) {
            key[r] = p.keys_in[base + idx];
            val[r] = p.vals_in ? p.vals_in[base + idx] : (uint32_t)(begin + idx);
            if (p.drop_culled) vld[r] = key[r] != 0xFFFFFFFFu;
        }
    }
#pragma unroll
    for (int r = 0; r < SORT_IPT; ++r) {
        const bool valid = vld[r];
        const uint32_t kk = key[r], vv = val[r];
        const uint32_t d = valid ? (kk >> p.shift) & p.mask : (uint32_t)RADIX;
        // lanes holding the same digit (or both invalid): the intersection of
        // nine ballots, one per bit of d (0..RADIX)
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < 9; ++b) {
            const bool set = ((d >> b) & 1u) != 0u;
            const unsigned bal = __ballot_sync(0xffffffffu, set);
            peers &= set ? bal : ~bal;
        }
        uint32_t before = 0;
        if (valid) before = s_wcnt[warp][d];
        __syncwarp();
        if (valid && (peers & lt) == 0) s_wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
        key[r] = kk;
        val[r] = vv;
        rank[r] = valid ? before + __popc(peers & lt) : 0xFFFFFFFFu;
    }
    __syncthreads();
    // thread d: prefix of digit d over warps, then block scan over digits
    uint32_t tot = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        uint32_t t = s_wcnt[w][threadIdx.x];
        s_wcnt[w][threadIdx.x] = tot;
        tot += t;
    }
    uint32_t nvalid;
    const uint32_t excl = block_excl_scan(tot, s_tmp, &nvalid);
    s_boff[threadIdx.x] = excl;
    s_goff[threadIdx.x] = p.hist[(int64_t)RADIX * p.chunk_base[s] + (int64_t)threadIdx.x * cps + k];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < SORT_IPT; ++r) {
        if (rank[r] != 0xFFFFFFFFu) {
            const uint32_t d = (key[r] >> p.shift) & p.mask;
            const uint32_t pos = s_boff[d] + s_wcnt[warp][d] + rank[r];
            s_key[pos] = key[r];
            s_val[pos] = val[r];
        }
    }
    __syncthreads();
    const int64_t obase = p.seg_off[s];
    for (int j = threadIdx.x; j < (int)nvalid; j += SORT_THREADS) {
        const uint32_t kk = s_key[j];
        const uint32_t d = (kk >> p.shift) & p.mask;
        const int64_t pos = obase + s_goff[d] + (uint32_t)(j - s_boff[d]);
        p.keys_out[pos] = kk;
        p.vals_out[pos] = s_val[j];
    }
}

cudaError_t launch_radix_pass(const RadixPass &p, cudaStream_t st)
{
    if (p.n_seg <= 0 || p.total_chunks <= 0) return cudaSuccess;
    k_radix_upsweep<<<p.total_chunks, SORT_THREADS, 0, st>>>(p);
    k_digit_scan<<<dim3(p.n_seg, RADIX / DSCAN_WARPS), 32 * DSCAN_WARPS, 0, st>>>(p.hist, p.dtot, p.chunk_base,
                                                                                   p.len_out);
    k_radix_scatter<<<p.total_chunks, SORT_THREADS, 0, st>>>(p);
    return cudaGetLastError();
}

// ------------------------------------------------------ K3 tile counts -----
// Each view's visible Gaussians, in depth order, are cut into chunks of
// cp.bin_chunk.  Per chunk, k_tile_count counts how many of them cover each
// tile: every rectangle adds +1/-1 at its four corners of a 2D difference
// array in shared memory, and two prefix sums (along x, then y) turn it into
// counts.  The tile grid is processed in row bands that fit shared memory.
// It also writes the rectangles in depth order (srect) for K4.
constexpr int BIN_THREADS = 256;

__global__ void __launch_bounds__(BIN_THREADS)
k_tile_count(const uint32_t *__restrict__ sorted_g, const uint32_t *__restrict__ n_vis,
             const uint2 *__restrict__ rect, Layout L, CamParams cp, int band_rows, uint2 *__restrict__ srect,
             uint32_t *__restrict__ bhist)
{
    extern __shared__ uint32_t s_d[];   // (band_rows + 1) x (ntx + 1)
    chain_wait();
    const int c = blockIdx.x;
    const int v = find_segment(L.cb_base, L.V, c);
    const int k = c - L.cb_base[v];
    const int64_t S = L.vd_off[v + 1] - L.vd_off[v];
    const int64_t nv = min64(n_vis[v], S);
    const int64_t begin = (int64_t)k * cp.bin_chunk;
    if (begin >= nv) return;
    const int n = (int)min64(cp.bin_chunk, nv - begin);
    const int ntx = cp.ntx, W = ntx + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t *g = sorted_g + L.vd_off[v] + begin;
    const uint2 *rv = rect + L.vd_off[v];
    uint2 *sr = srect + L.vd_off[v] + begin;
    uint32_t *h = bhist + (int64_t)cp.n_tiles * c;
    for (int r0 = 0; r0 < cp.nty; r0 += band_rows) {
        const int r1 = min(cp.nty, r0 + band_rows), H = r1 - r0;
        for (int i = threadIdx.x; i < (H + 1) * W; i += BIN_THREADS) s_d[i] = 0;
        __syncthreads();
        for (int j = threadIdx.x; j < n; j += BIN_THREADS) {
            uint2 rc;
            if (r0 == 0) {               // first band: gather in depth order
                rc = rv[g[j]];
                sr[j] = rc;
            } else {
                rc = sr[j];              // written by this thread in band 0
            }
            const int y0 = (int)(rc.y & 0xFFFFu), y1 = (int)(rc.y >> 16);
            if (y1 < r0 || y0 >= r1) continue;
            const int x0 = (int)(rc.x & 0xFFFFu), x1 = (int)(rc.x >> 16);
            const int ya = max(y0, r0) - r0, yb = min(y1, r1 - 1) - r0 + 1;
            atomicAdd(&s_d[ya * W + x0], 1u);
            atomicAdd(&s_d[ya * W + x1 + 1], 0xFFFFFFFFu);
            atomicAdd(&s_d[yb * W + x0], 0xFFFFFFFFu);
            atomicAdd(&s_d[yb * W + x1 + 1], 1u);
        }
        __syncthreads();
        for (int y = warp; y < H; y += BIN_THREADS / 32) {      // prefix along x: a warp per row
            uint32_t carry = 0;
            for (int x0 = 0; x0 < ntx; x0 += 32) {
                const int x = x0 + lane;
                uint32_t inc = x < ntx ? s_d[y * W + x] : 0u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += t;
                }
                if (x < ntx) s_d[y * W + x] = carry + inc;
                carry += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
        __syncthreads();
        for (int x = threadIdx.x; x < ntx; x += BIN_THREADS) {  // prefix along y: a thread per column
            uint32_t run = 0;
            for (int y = 0; y < H; ++y) {
                run += s_d[y * W + x];
                s_d[y * W + x] = run;
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < H * ntx; t += BIN_THREADS) {
            const int y = t / ntx, x = t - y * ntx;
            h[(int64_t)r0 * ntx + t] = s_d[y * W + x];
        }
        __syncthreads();
    }
}

// Per view: bhist[chunk][tile] becomes the exclusive prefix over the view's
// chunks (each chunk's first slot inside a tile's list, relative to the
// tile's start), totals -> ranges[v][tile].y; then the view's last block to
// finish scans the totals in tile order into ranges[v][tile] = [begin, end)
// (empty tiles [0, 0)) and n_inst[v], and lists the heavy tiles for the blend
// (two launches less than with kernels of their own).  The chunk prefix: a block
// per (view, 32 tiles), SEGS threads per tile, each holding up to TCOL_SEG of the
// tile's chunks in registers (all its loads in flight at once), so a view's ~80
// chunks are scanned as eight short runs plus a prefix over the eight run totals,
// and the hundreds of smaller chunks of a call of few views as 32 runs.
constexpr int TCOL_TILES = 32;
constexpr int TCOL_SEG = 16;                         // chunks per run in registers
constexpr int TSCAN_PER = 4;                         // tiles per thread and round of the final scan

template <int SEGS>
__global__ void __launch_bounds__(TCOL_TILES * SEGS, SEGS > 8 ? 1 : 4)
k_tile_chunk_scan(const uint32_t *__restrict__ n_vis, Layout L, CamParams cp, uint32_t *__restrict__ bhist,
                  int2 *ranges, uint32_t *__restrict__ n_inst, int *__restrict__ done, int *__restrict__ overflow,
                  BlendQueue queue)
{
    constexpr int NT = TCOL_TILES * SEGS;
    __shared__ uint32_t s_run[SEGS][TCOL_TILES];
    __shared__ uint32_t s_tmp[33];
    __shared__ int s_last;
    chain_wait();
    const int v = blockIdx.y;
    const int tl = threadIdx.x % TCOL_TILES, sg = threadIdx.x / TCOL_TILES;
    const int t = blockIdx.x * TCOL_TILES + tl;
    const int nt = cp.n_tiles;
    const int64_t S = L.vd_off[v + 1] - L.vd_off[v];
    const int64_t nv = min64(n_vis[v], S);
    const int nch = (int)ceil_div(nv, cp.bin_chunk);
    uint32_t *h = bhist + (int64_t)nt * L.cb_base[v] + t;
    int2 *const R = ranges + (int64_t)v * nt;
    const int per = (int)ceil_div(nch, SEGS);           // chunks of this thread's run
    const int c0 = min(nch, sg * per), c1 = min(nch, c0 + per);
    const int m = t < nt ? c1 - c0 : 0;
    uint32_t *hp = h + (int64_t)c0 * nt;
    uint32_t sum = 0, x[TCOL_SEG];
    if (per <= TCOL_SEG) {                              // uniform over the block
#pragma unroll
        for (int j = 0; j < TCOL_SEG; ++j) x[j] = j < m ? hp[(int64_t)j * nt] : 0u;
#pragma unroll
        for (int j = 0; j < TCOL_SEG; ++j) sum += x[j];
    } else {                                            // views of more than SEGS * TCOL_SEG chunks
        for (int j = 0; j < m; ++j) sum += hp[(int64_t)j * nt];
    }
    s_run[sg][tl] = sum;
    __syncthreads();
    uint32_t run = 0;
    for (int k = 0; k < sg; ++k) run += s_run[k][tl];
    if (per <= TCOL_SEG) {
#pragma unroll
        for (int j = 0; j < TCOL_SEG; ++j)
            if (j < m) {
                hp[(int64_t)j * nt] = run;
                run += x[j];
            }
    } else {
        for (int j = 0; j < m; ++j) {
            const uint32_t y = hp[(int64_t)j * nt];
            hp[(int64_t)j * nt] = run;
            run += y;
        }
    }
    if (sg == SEGS - 1 && t < nt) __stcg(&R[t].y, (int)run);
    // the view's last block scans the totals of all its tiles
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done + v, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    uint32_t carry = 0;
    for (int t0 = 0; t0 < nt; t0 += NT * TSCAN_PER) {
        const int a = t0 + (int)threadIdx.x * TSCAN_PER;
        uint32_t y[TSCAN_PER], mine = 0, tot;
#pragma unroll
        for (int j = 0; j < TSCAN_PER; ++j) {
            y[j] = a + j < nt ? (uint32_t)__ldcg(&R[a + j].y) : 0u;
            mine += y[j];
        }
        uint32_t at = carry + block_excl_scan(mine, s_tmp, &tot);
#pragma unroll
        for (int j = 0; j < TSCAN_PER; ++j) {
            if (a + j >= nt) break;
            R[a + j] = y[j] ? make_int2((int)at, (int)(at + y[j])) : make_int2(0, 0);
            if (queue.count && y[j] >= (uint32_t)BLEND_HEAVY) queue.list[atomicAdd(queue.count + 1, 1)] = v * nt + a + j;
            at += y[j];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        n_inst[v] = carry;
        if ((int64_t)carry > L.io_off[v + 1] - L.io_off[v]) atomicExch(overflow, 1);
    }
}

cudaError_t launch_tile_count(const uint32_t *sorted_g, const uint32_t *n_vis, const uint2 *rect, const Layout &L,
                              const CamParams &cp, int n_chunks, int view_chunks, uint2 *srect, uint32_t *bhist,
                              int2 *ranges, uint32_t *n_inst, int *done, int *overflow, BlendQueue queue,
                              cudaStream_t st)
{
    if (L.V <= 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (n_chunks > 0) {
        const int W = cp.ntx + 1;
        const int band_rows = max(1, min(cp.nty, TILE_COUNT_SMEM / (4 * W) - 1));
        const size_t smem = 4 * (size_t)(band_rows + 1) * W;
        e = launch_chained(k_tile_count, dim3(n_chunks), dim3(BIN_THREADS), smem, st, 1, sorted_g, n_vis, rect, L, cp,
                           band_rows, srect, bhist);
        if (e != cudaSuccess) return e;
    }
    const dim3 cgrid((unsigned)ceil_div(cp.n_tiles, TCOL_TILES), L.V);
    // by the chunks a view may have; about a third of them hold visible Gaussians,
    // and the wide form costs the 64 views of 157 chunks 48 us more (147 for 99 us)
    if (view_chunks <= 4 * 8 * TCOL_SEG)
        return launch_chained(k_tile_chunk_scan<8>, cgrid, dim3(TCOL_TILES * 8), 0, st, 1, n_vis, L, cp, bhist, ranges,
                              n_inst, done, overflow, queue);
    return launch_chained(k_tile_chunk_scan<32>, cgrid, dim3(TCOL_TILES * 32), 0, st, 1, n_vis, L, cp, bhist, ranges,
                          n_inst, done, overflow, queue);
}

// ------------------------------------------------------ K4 tile emission ----
// A warp per (chunk, tile row).  The block stages the chunk's depth-ordered
// (rectangle, Gaussian) pairs in shared memory; each warp picks, in order,
// the pairs whose rectangle covers its row (into a per-warp queue of pair
// indices) and writes every queued pair into each covered tile's list at that
// tile's running slot.  The pairs are taken
// in depth order, so every list comes out ordered by (depth, index) without a
// sort over the instances.
//
// k_tile_emit_flat: rows of at most EMIT_FLAT_MAX_NTX tiles.  32 queued pairs
// are written at a time with no loop over tiles or column bands: queued pair
// e (lane e) XORs its lane bit into a difference array along the row at x0
// and at x1 + 1, so the array's inclusive XOR prefix is, for every tile x,
// the mask M[x] of the queued pairs covering x.  Pair e's slot in tile x is
// cnt[x] + popc(M[x] & bits below e) -- its rank among the chunk's pairs
// covering x, in depth order -- so the instances can be written in any order
// (lane e writes its pair's first EMIT_JCAP columns; the columns of wider
// spans are spread over the lanes), and then cnt[x] += popc(M[x]).
// k_tile_emit_smem: any row width, slots in shared memory, a lane per
// column of each queued pair.
constexpr int EMIT_STAGE = BIN_CHUNK_MAX;             // a whole chunk of the usual size: one barrier
constexpr int EMIT_FLAT_MAX_NTX = 256;
constexpr int EMIT_STEP = 512;                        // pairs a warp queues at a time: a 16-bit half word a lane
constexpr int EMIT_Q = 31 + EMIT_STEP;                // queue entries per warp
constexpr int EMIT_WORDS = EMIT_STAGE / 32;           // words of a row's bits
constexpr int EMIT_JCAP = 4;                          // columns a pair's own lane writes
constexpr int EMIT_DYN_MIN_CHUNKS = 1024;             // about a full wave of eight-warp blocks

struct EmitChunk {
    int v, n;
    int64_t begin, nv;
    bool skip;
};

__device__ __forceinline__ EmitChunk emit_chunk(const uint32_t *n_vis, const uint32_t *n_inst, const Layout &L,
                                                const CamParams &cp)
{
    EmitChunk ch;
    const int c = blockIdx.x;
    ch.v = find_segment(L.cb_base, L.V, c);
    const int k = c - L.cb_base[ch.v];
    const int64_t S = L.vd_off[ch.v + 1] - L.vd_off[ch.v];
    const int64_t nv = min64(n_vis[ch.v], S);
    ch.nv = nv;
    ch.begin = (int64_t)k * cp.bin_chunk;
    ch.skip = ch.begin >= nv ||                                             // past the visible list
              (int64_t)n_inst[ch.v] > L.io_off[ch.v + 1] - L.io_off[ch.v];   // overflow: nothing emitted
    ch.n = ch.skip ? 0 : (int)min64(cp.bin_chunk, nv - ch.begin);
    return ch;
}

// RMASK (grids of at most 32 tile rows): the stage turns the pairs' row masks, 32 at a
// time, into the rows' pair masks (a bit transpose by shuffles), so a warp reads its
// row's pairs as words of bits instead of testing every pair of the chunk against the
// row: 54.7M instructions for 16 driving views instead of 72.5M, 64 views 358 -> 334
// us.  What is left waits: a chunk's heaviest row keeps its block alive (the SMs idle
// 29% of the 16 views' launch), and the chain from queue to slot to store.
// DYN (with RMASK, chunks of at most one stage): one block per chunk, whose
// warps take the chunk's rows from a counter, heaviest row first (the row
// through the horizon holds several times the average row's instances, and
// a block of fixed rows lives as long as its heaviest one).  Otherwise a
// block per (chunk, 8 rows), a warp per row.
template <int CPL, bool RMASK, bool DYN>
__global__ void __launch_bounds__(TILE_EMIT_WARPS * 32, 6)
k_tile_emit_flat(const uint32_t *__restrict__ sorted_g, const uint2 *__restrict__ srect,
                 const uint32_t *__restrict__ n_vis, const uint32_t *__restrict__ n_inst,
                 const uint32_t *__restrict__ bhist, const int2 *__restrict__ ranges, Layout L, CamParams cp,
                 uint32_t *__restrict__ inst_gauss)
{
    static_assert(CPL % 4 == 0, "columns per lane in 16-byte groups");
    static_assert(!DYN || RMASK, "dynamic rows need the 32-row mask");
    constexpr int NC = 32 * CPL;                        // columns a warp's arrays hold (>= ntx)
    __shared__ uint32_t s_y[EMIT_STAGE];                // RMASK: bits [row][pair], else y0 | y1 << 16
    __shared__ uint16_t s_x[EMIT_STAGE];                // x0 | x1 << 8 (rows of at most 256 tiles)
    __shared__ uint32_t s_g[EMIT_STAGE];
    __shared__ uint16_t s_q[TILE_EMIT_WARPS][EMIT_Q];   // staged-pair indices
    __shared__ __align__(16) uint32_t s_cnt[TILE_EMIT_WARPS][NC];
    __shared__ __align__(16) uint32_t s_m[TILE_EMIT_WARPS][NC + 4];   // x1 + 1 <= ntx <= NC
    __shared__ uint32_t s_load[32];                     // DYN: the chunk's instances per row
    __shared__ int s_order[32];                         // DYN: rows, heaviest first
    __shared__ int s_next;
    chain_wait();
    const EmitChunk ch = emit_chunk(n_vis, n_inst, L, cp);
    if (ch.skip) return;
    const int v = ch.v, n = ch.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ntx = cp.ntx;
    uint16_t *q = s_q[warp];
    uint32_t *out = inst_gauss + L.io_off[v];
    uint32_t *cnt = s_cnt[warp];
    uint32_t *M = s_m[warp];
    const uint32_t *hc = bhist + (int64_t)cp.n_tiles * blockIdx.x;
    const int2 *Rv = ranges + (int64_t)v * cp.n_tiles;
    const unsigned lt = lanemask_lt();
    int head = 0, tail = 0;                             // queued: [head, tail)
    // slot counters of a row: the tiles' list starts plus the chunk's offsets
    auto init_row = [&](int row) {
        const uint32_t *h = hc + (int64_t)row * ntx;
        const int2 *R = Rv + (int64_t)row * ntx;
        for (int x = lane; x < NC; x += 32) cnt[x] = x < ntx ? (uint32_t)R[x].x + h[x] : 0u;
        for (int x = lane; x < NC + 4; x += 32) M[x] = 0u;
    };
    // writes the ne (1..32) pairs at the head of the queue
    auto drain = [&](int ne) {
        __syncwarp();
        uint32_t gv = 0u;
        int x0 = 0, w = 0;
        if (lane < ne) {
            const int i = q[head + lane];
            const uint32_t xs = s_x[i];
            gv = s_g[i];
            x0 = (int)(xs & 0xFFu);
            w = (int)(xs >> 8) - x0 + 1;
            atomicXor(&M[x0], 1u << lane);
            atomicXor(&M[x0 + w], 1u << lane);
        }
        head += ne;
        __syncwarp();
        // inclusive XOR prefix along the row: lane l holds columns CPL l ..
        // CPL l + CPL - 1 in registers, one warp scan of the lanes' totals
        uint32_t m[CPL];
#pragma unroll
        for (int k = 0; k < CPL; k += 4) {
            const uint4 t = *reinterpret_cast<const uint4 *>(M + CPL * lane + k);
            m[k] = t.x; m[k + 1] = t.y; m[k + 2] = t.z; m[k + 3] = t.w;
        }
#pragma unroll
        for (int k = 1; k < CPL; ++k) m[k] ^= m[k - 1];
        uint32_t inc = m[CPL - 1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc ^= t;
        }
        const uint32_t ex = inc ^ m[CPL - 1];
#pragma unroll
        for (int k = 0; k < CPL; k += 4) {
            m[k] ^= ex; m[k + 1] ^= ex; m[k + 2] ^= ex; m[k + 3] ^= ex;
            *reinterpret_cast<uint4 *>(M + CPL * lane + k) = make_uint4(m[k], m[k + 1], m[k + 2], m[k + 3]);
        }
        __syncwarp();
        const int wl = min(w, EMIT_JCAP);
        for (int j = 0; j < wl; ++j) {
            const int x = x0 + j;
            out[cnt[x] + __popc(M[x] & lt)] = gv;
        }
        // columns past EMIT_JCAP: instance I of the concatenated remainders
        // belongs to the pair whose inclusive prefix first exceeds I
        const int rw = max(w - EMIT_JCAP, 0);
        if (__any_sync(0xffffffffu, rw > 0)) {
            int incl = rw;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            for (int base = 0; base < total; base += 32) {
                const int I = base + lane;
                int e = 0;                              // the number of pairs with incl <= I
#pragma unroll
                for (int s = 16; s > 0; s >>= 1) {
                    const int t = __shfl_sync(0xffffffffu, incl, e + s - 1);
                    if (t <= I) e += s;
                }
                const int start = __shfl_sync(0xffffffffu, incl - rw, e);
                const int xe = __shfl_sync(0xffffffffu, x0, e);
                const uint32_t ge = __shfl_sync(0xffffffffu, gv, e);
                if (I < total) {
                    const int x = xe + EMIT_JCAP + (I - start);
                    out[cnt[x] + __popc(M[x] & ((1u << e) - 1u))] = ge;
                }
            }
        }
        __syncwarp();
        // cnt[x] += popc(M[x]) from the registers; M back to zero
#pragma unroll
        for (int k = 0; k < CPL; k += 4) {
            uint4 c = *reinterpret_cast<const uint4 *>(cnt + CPL * lane + k);
            c.x += __popc(m[k]); c.y += __popc(m[k + 1]); c.z += __popc(m[k + 2]); c.w += __popc(m[k + 3]);
            *reinterpret_cast<uint4 *>(cnt + CPL * lane + k) = c;
            *reinterpret_cast<uint4 *>(M + CPL * lane + k) = make_uint4(0u, 0u, 0u, 0u);
        }
        if (lane == 0) M[NC] = 0u;
        __syncwarp();
    };
    // one row over the m staged pairs: the row's bits, 512 pairs a step and 16 a lane,
    // become queue entries in pair order (a warp scan of the lanes' counts), written
    // out 32 at a time and emptied at the end (before the stage is replaced; one call
    // site of the drain)
    auto scan_row = [&](int row, int m) {
        int i0 = 0;
        while (true) {
            const int qn = tail - head;                 // at most 31 + 512
            if (qn >= 32 || (i0 >= m && qn > 0)) {
                drain(min(qn, 32));
                continue;
            }
            if (i0 >= m) break;
            if (head > 0) {                             // fewer than 32 left: to the front
                const uint16_t t = lane < qn ? q[head + lane] : (uint16_t)0;
                __syncwarp();
                if (lane < qn) q[lane] = t;
                head = 0;
                tail = qn;
            }
            const int base = i0 + 16 * lane;            // pairs base .. base + 15 are this lane's
            uint32_t bits = 0u;
            if (RMASK) {
                if (base < m) bits = s_y[row * EMIT_WORDS + ((base / 32 + row) & (EMIT_WORDS - 1))];
            } else {
                const int words = min(EMIT_STEP / 32, (m - i0 + 31) / 32);
                for (int k = 0; k < words; ++k) {
                    const int i = i0 + 32 * k + lane;
                    const uint32_t y = i < m ? s_y[i] : 0xFFFFu;              // y0 > y1: no row
                    const unsigned b = __ballot_sync(0xffffffffu, (int)(y & 0xFFFFu) <= row && row <= (int)(y >> 16));
                    if (lane >> 1 == k) bits = b;
                }
            }
            bits = (bits >> (base & 16)) & 0xFFFFu;
            int inc = __popc(bits);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            int at = tail + inc - __popc(bits);
            for (; bits; bits &= bits - 1u) q[at++] = (uint16_t)(base + __ffs(bits) - 1);
            tail += __shfl_sync(0xffffffffu, inc, 31);
            i0 += EMIT_STEP;
        }
        head = tail = 0;
    };
    const uint32_t *g = sorted_g + L.vd_off[v] + ch.begin;
    const uint2 *sr = srect + L.vd_off[v] + ch.begin;
    auto stage = [&](int s0, int m) {
        // whole warps: 32 pairs a warp's round
        for (int j0 = 32 * warp; j0 < m; j0 += TILE_EMIT_WARPS * 32) {
            const int j = j0 + lane;
            uint2 rc = make_uint2(0u, 0u);
            if (j < m) {
                rc = sr[s0 + j];
                s_x[j] = (uint16_t)((rc.x & 0xFFu) | rc.x >> 16 << 8);
                s_g[j] = g[s0 + j];
            }
            if (RMASK) {
                const uint32_t y0 = rc.y & 0xFFFFu, y1 = rc.y >> 16;     // y0 <= y1 <= 31
                uint32_t b = j < m ? ((2u << y1) - 1u) & (0xFFFFFFFFu << y0) : 0u;
                // 32 x 32 bit transpose: from a pair's rows to a row's pairs, by halves
                uint32_t low = 0x0000FFFFu;             // bits k with (k & o) == 0
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const uint32_t t = __shfl_xor_sync(0xffffffffu, b, o);
                    b = lane & o ? (b & ~low) | ((t & ~low) >> o) : (b & low) | ((t & low) << o);
                    low ^= low << (o >> 1);
                }
                // rows shifted by one bank each: no conflict across rows or along them
                s_y[lane * EMIT_WORDS + ((j0 / 32 + lane) & (EMIT_WORDS - 1))] = b;
            } else if (j < m) {
                s_y[j] = rc.y;
            }
        }
    };
    if (DYN) {
        const int nty = cp.nty;                         // <= 32; n <= EMIT_STAGE
        if (threadIdx.x < 32) s_load[threadIdx.x] = 0u;
        if (threadIdx.x == 0) s_next = 0;
        stage(0, n);
        __syncthreads();
        // the chunk's instances per row: its tiles' offsets up to the next
        // chunk's (the exclusive prefix over the view's chunks), or up to the
        // tile's total for the view's last chunk
        const bool last = ch.begin + cp.bin_chunk >= ch.nv;
        for (int t = threadIdx.x; t < nty * ntx; t += TILE_EMIT_WARPS * 32) {
            const uint32_t nxt = last ? (uint32_t)(Rv[t].y - Rv[t].x) : hc[(int64_t)cp.n_tiles + t];
            const uint32_t c = nxt - hc[t];
            if (c) atomicAdd(&s_load[t / ntx], c);
        }
        __syncthreads();
        if (warp == 0) {                                // heaviest row first, ties by row
            const uint32_t ld = lane < nty ? s_load[lane] : 0u;
            int rank = 0;
            for (int k = 0; k < nty; ++k) {
                const uint32_t o = __shfl_sync(0xffffffffu, ld, k);
                rank += (o > ld || (o == ld && k < lane)) ? 1 : 0;
            }
            if (lane < nty) s_order[rank] = lane;
        }
        __syncthreads();
        while (true) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&s_next, 1);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k >= nty) break;
            const int row = s_order[k];
            init_row(row);
            scan_row(row, n);
        }
    } else {
        const int row = blockIdx.y * TILE_EMIT_WARPS + warp;
        const bool active = row < cp.nty;
        if (active) init_row(row);
        for (int s0 = 0; s0 < n; s0 += EMIT_STAGE) {
            const int m = min(EMIT_STAGE, n - s0);
            __syncthreads();
            stage(s0, m);
            __syncthreads();
            if (active) scan_row(row, m);
        }
    }
}

__global__ void __launch_bounds__(TILE_EMIT_WARPS * 32)
k_tile_emit_smem(const uint32_t *__restrict__ sorted_g, const uint2 *__restrict__ srect,
                 const uint32_t *__restrict__ n_vis, const uint32_t *__restrict__ n_inst,
                 const uint32_t *__restrict__ bhist, const int2 *__restrict__ ranges, Layout L, CamParams cp,
                 uint32_t *__restrict__ inst_gauss)
{
    __shared__ uint2 s_rc[EMIT_STAGE];
    __shared__ uint32_t s_g[EMIT_STAGE];
    __shared__ uint2 s_q[TILE_EMIT_WARPS][64];
    extern __shared__ uint32_t s_cnt[];                 // [TILE_EMIT_WARPS][ntx]
    chain_wait();
    const EmitChunk ch = emit_chunk(n_vis, n_inst, L, cp);
    if (ch.skip) return;
    const int v = ch.v, n = ch.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = blockIdx.y * TILE_EMIT_WARPS + warp;
    const bool active = row < cp.nty;
    const int ntx = cp.ntx;
    uint2 *q = s_q[warp];
    uint32_t *out = inst_gauss + L.io_off[v];
    uint32_t *cnt = s_cnt + warp * ntx;
    if (active) {
        const uint32_t *h = bhist + (int64_t)cp.n_tiles * blockIdx.x + (int64_t)row * ntx;
        const int2 *R = ranges + (int64_t)v * cp.n_tiles + (int64_t)row * ntx;
        for (int x = lane; x < ntx; x += 32) cnt[x] = (uint32_t)R[x].x + h[x];
    }
    auto drain = [&](int cnt_q) {
        for (int j = 0; j < cnt_q; ++j) {
            const uint2 e = q[j];
            const uint32_t x0 = e.y & 0xFFFFu, x1 = e.y >> 16;
            for (uint32_t x = x0 + (((uint32_t)lane - x0) & 31u); x <= x1; x += 32) {
                const uint32_t p = cnt[x];
                out[p] = e.x;
                cnt[x] = p + 1;
            }
        }
    };
    const uint32_t *g = sorted_g + L.vd_off[v] + ch.begin;
    const uint2 *sr = srect + L.vd_off[v] + ch.begin;
    const unsigned lt = lanemask_lt();
    int qn = 0;
    for (int s0 = 0; s0 < n; s0 += EMIT_STAGE) {
        const int m = min(EMIT_STAGE, n - s0);
        __syncthreads();
        for (int j = threadIdx.x; j < m; j += TILE_EMIT_WARPS * 32) {
            s_rc[j] = sr[s0 + j];
            s_g[j] = g[s0 + j];
        }
        __syncthreads();
        if (!active) continue;
        for (int i0 = 0; i0 < m; i0 += 32) {
            const int i = i0 + lane;
            bool p = false;
            uint2 e = make_uint2(0u, 0u);
            if (i < m) {
                const uint2 rc = s_rc[i];
                p = (int)(rc.y & 0xFFFFu) <= row && row <= (int)(rc.y >> 16);
                e = make_uint2(p ? s_g[i] : 0u, rc.x);
            }
            const unsigned mask = __ballot_sync(0xffffffffu, p);
            if (p) q[qn + __popc(mask & lt)] = e;
            qn += __popc(mask);
            if (qn >= 32) {
                __syncwarp();
                drain(qn);
                qn = 0;
                __syncwarp();
            }
        }
    }
    if (active && qn > 0) {
        __syncwarp();
        drain(qn);
    }
}

cudaError_t launch_tile_emit(const uint32_t *sorted_g, const uint2 *srect, const uint32_t *n_vis,
                             const uint32_t *n_inst, const uint32_t *bhist, const int2 *ranges, const Layout &L,
                             const CamParams &cp, int n_chunks, uint32_t *inst_gauss, cudaStream_t st)
{
    if (n_chunks <= 0 || L.V <= 0) return cudaSuccess;
    const dim3 grid(n_chunks, (unsigned)ceil_div(cp.nty, TILE_EMIT_WARPS));
    // a block per chunk needs enough chunks to fill the GPU (a one-view launch
    // has ~80); fewer take a block per (chunk, eight rows)
    const bool rm = cp.nty <= 32, dyn = rm && cp.bin_chunk <= EMIT_STAGE && n_chunks >= EMIT_DYN_MIN_CHUNKS;
    const dim3 grid1(n_chunks, 1);
    const dim3 block(TILE_EMIT_WARPS * 32);
#define EMIT_FLAT(CPL_)                                                                                         \
    return dyn  ? launch_chained(k_tile_emit_flat<CPL_, true, true>, grid1, block, 0, st, 1, sorted_g, srect,    \
                                 n_vis, n_inst, bhist, ranges, L, cp, inst_gauss)                               \
           : rm ? launch_chained(k_tile_emit_flat<CPL_, true, false>, grid, block, 0, st, 1, sorted_g, srect,    \
                                 n_vis, n_inst, bhist, ranges, L, cp, inst_gauss)                               \
                : launch_chained(k_tile_emit_flat<CPL_, false, false>, grid, block, 0, st, 1, sorted_g, srect,   \
                                 n_vis, n_inst, bhist, ranges, L, cp, inst_gauss)
    if (cp.ntx <= 128) EMIT_FLAT(4);
    if (cp.ntx <= EMIT_FLAT_MAX_NTX) EMIT_FLAT(8);
#undef EMIT_FLAT
    const size_t smem = 4 * (size_t)TILE_EMIT_WARPS * cp.ntx;
    return launch_chained(k_tile_emit_smem, grid, block, smem, st, 1, sorted_g, srect, n_vis, n_inst, bhist, ranges, L, cp,
                          inst_gauss);
}

cudaError_t configure_sort_kernels()
{
    cudaError_t e = cudaFuncSetAttribute(k_depth_sort<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_depth_sort<32>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    if (depth_sort_cluster<16>() <= 0 || depth_sort_cluster<32>() <= 0) return cudaErrorInvalidConfiguration;
    return cudaFuncSetAttribute(k_tile_emit_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, TILE_EMIT_SMEM_MAX);
}

// Tile id of every instance of one view, from its ranges (debug export).
__global__ void k_fill_tiles(const int2 *__restrict__ R, int n_tiles, uint32_t *__restrict__ tiles)
{
    const int t = blockIdx.x;
    if (t >= n_tiles) return;
    const int2 r = R[t];
    for (int j = r.x + threadIdx.x; j < r.y; j += blockDim.x) tiles[j] = (uint32_t)t;
}

cudaError_t launch_fill_tiles(const int2 *ranges_view, int n_tiles, uint32_t *tiles_view, cudaStream_t st)
{
    if (n_tiles <= 0) return cudaSuccess;
    k_fill_tiles<<<n_tiles, 128, 0, st>>>(ranges_view, n_tiles, tiles_view);
    return cudaGetLastError();
}

}  // namespace reloc
