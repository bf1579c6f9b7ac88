// Grouping of samples by cluster label: the cluster set S of Alg. 1/3 as a
// CSR (offsets[k + 1], members[n]) with the members of each cluster in
// ascending sample id.  Built as a stable LSD radix sort of the labels whose
// values are the sample ids.
//
// A pass moves up to 10 bits, the bits of k shared out evenly (k < 1,024: one
// pass; k < 2^20: two), and is three launches: every block counts the digits
// of its share of the elements (k_radix_hist), a warp per digit turns the
// blocks' counts into starts (k_radix_cols), and every block ranks and moves
// its elements (k_radix_scatter).  The grid is at most GR_BLOCKS blocks, each
// walking consecutive tiles with running starts, so the table of counts stays
// small (at most 1,024 x 1,216) and needs no scan of its own over tiles.  With one pass
// the digits are the labels and their starts the offsets; otherwise
// k_group_offsets finds each cluster's start in the sorted keys.
//
// Launches bound this step: 8-bit digits, a table per tile with three scan
// launches a pass, and a label histogram with its own scan took 15 launches
// and 69 us at 300,000 samples, k = 3,000; these 7 take 35 us (a tile's
// ranking chain is about 6 us of each scatter, so tiles are small and the
// blocks many).
#include "common.cuh"

namespace gkm {

constexpr int GR_BITS = 10;            // widest digit
constexpr int GR_BINS = 1 << GR_BITS;
constexpr int GR_THREADS = 256;
constexpr int GR_WARPS = GR_THREADS / 32;
constexpr int GR_ITEMS = 8;            // elements per thread and tile; a warp owns GR_ITEMS * 32 consecutive ones
constexpr int GR_TILE = GR_THREADS * GR_ITEMS;
constexpr int GR_BLOCKS = 1216;        // eight blocks per SM

// The sort key of a label: a label outside [0, k) sorts as k, after every
// cluster, so that it cannot shift the member ranges of the valid clusters
// (it belongs to no cluster and is recorded in the status word).  The passes
// cover the bits of k itself for this reason.
__device__ __forceinline__ int32_t sort_key(int32_t label, int32_t k)
{
    return (uint32_t)label < (uint32_t)k ? label : k;
}

// Digits of a block's tiles [t0, t1), into hist[digit * gridDim.x + block].  The first pass (st given) records labels
// out of range.  zero: a counter cleared for a later kernel of the caller (may be NULL).
__global__ void __launch_bounds__(GR_THREADS) k_radix_hist(const int32_t *__restrict__ keys, int64_t n, int32_t k,
                                                           int shift, int bins, int64_t tiles_per_block,
                                                           int32_t *__restrict__ hist, DevStatus *st,
                                                           unsigned *__restrict__ zero)
{
    __shared__ int h[GR_BINS];
    for (int b = threadIdx.x; b < bins; b += GR_THREADS)
        h[b] = 0;
    if (zero && blockIdx.x == 0 && threadIdx.x == 0)
        *zero = 0u;
    __syncthreads();
    const int64_t e0 = blockIdx.x * tiles_per_block * GR_TILE, e1 = min(n, e0 + tiles_per_block * GR_TILE);
#pragma unroll 4
    for (int64_t e = e0 + threadIdx.x; e < e1; e += GR_THREADS) {
        const int32_t label = keys[e];
        if (st && (uint32_t)label >= (uint32_t)k)
            flag_error(st, GK_ERR_INVALID, (unsigned)e);
        atomicAdd(&h[(sort_key(label, k) >> shift) & (bins - 1)], 1);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < bins; b += GR_THREADS)
        hist[(int64_t)b * gridDim.x + blockIdx.x] = h[b];
}

// One warp per digit: the blocks' counts to starts within the digit, in place, and the digit's total.
__global__ void __launch_bounds__(GR_THREADS) k_radix_cols(int32_t *__restrict__ hist, int nblocks, int bins,
                                                           int32_t *__restrict__ total)
{
    const int b = blockIdx.x * GR_WARPS + (threadIdx.x >> 5), lane = lane_id();
    if (b >= bins)
        return;
    int32_t *row = hist + (int64_t)b * nblocks;
    int carry = 0;
    for (int c0 = 0; c0 < nblocks; c0 += 32) {
        const int c = c0 + lane;
        const int v = c < nblocks ? row[c] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL_MASK, incl, o);
            if (lane >= o)
                incl += u;
        }
        if (c < nblocks)
            row[c] = carry + incl - v;
        carry += __shfl_sync(FULL_MASK, incl, 31);
    }
    if (lane == 0)
        total[b] = carry;
}

// Moves a block's elements to their places.  offsets (one pass only, may be NULL): the digits' starts are the
// clusters', written by block 0 with the counts (may be NULL).
__global__ void __launch_bounds__(GR_THREADS) k_radix_scatter(const int32_t *__restrict__ keys_in,
                                                              const int32_t *__restrict__ vals_in, int64_t n,
                                                              int32_t k, int shift, int bins, int64_t tiles_per_block,
                                                              const int32_t *__restrict__ hist,
                                                              const int32_t *__restrict__ total,
                                                              int32_t *__restrict__ keys_out,
                                                              int32_t *__restrict__ vals_out,
                                                              int32_t *__restrict__ offsets,
                                                              int32_t *__restrict__ counts)
{
    constexpr int PER = GR_BINS / GR_THREADS;  // digits per thread
    __shared__ int start[GR_BINS];             // next place of each digit for this block
    __shared__ unsigned short whist[GR_WARPS][GR_BINS];
    __shared__ int wsum[GR_WARPS];
    const int tid = threadIdx.x, w = tid >> 5, lane = lane_id();
    // starts of the digits: exclusive scan of the totals (thread t: digits PER t .. PER t + PER - 1)
    int tot[PER], sum = 0;
#pragma unroll
    for (int q = 0; q < PER; q++) {
        tot[q] = PER * tid + q < bins ? total[PER * tid + q] : 0;
        sum += tot[q];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o)
            incl += u;
    }
    if (lane == 31)
        wsum[w] = incl;
    __syncthreads();
    int at = incl - sum;
    for (int q = 0; q < w; q++)
        at += wsum[q];
#pragma unroll
    for (int q = 0; q < PER; q++) {
        const int b = PER * tid + q;
        if (b < bins) {
            start[b] = at + hist[(int64_t)b * gridDim.x + blockIdx.x];
            if (offsets && blockIdx.x == 0) {
                if (b <= k)
                    offsets[b] = at;  // b == k: where the labels out of range begin
                if (counts && b < k)
                    counts[b] = tot[q];
            }
        }
        at += tot[q];
    }
    for (int64_t t = blockIdx.x * tiles_per_block; t < (blockIdx.x + 1) * tiles_per_block && t * GR_TILE < n; t++) {
        for (int b = tid; b < GR_WARPS * GR_BINS / 2; b += GR_THREADS)
            reinterpret_cast<unsigned *>(&whist[0][0])[b] = 0u;
        __syncthreads();
        const int64_t wbase = t * GR_TILE + (int64_t)w * (GR_ITEMS * 32);
        int key[GR_ITEMS], val[GR_ITEMS], rank[GR_ITEMS];
#pragma unroll
        for (int r = 0; r < GR_ITEMS; r++) {
            const int64_t e = wbase + r * 32 + lane;
            key[r] = e < n ? sort_key(keys_in[e], k) : -1;
            val[r] = e < n ? (vals_in ? vals_in[e] : (int)e) : 0;
        }
#pragma unroll
        for (int r = 0; r < GR_ITEMS; r++) {
            const int dg = key[r] < 0 ? GR_BINS : (key[r] >> shift) & (bins - 1);
            const unsigned peers = __match_any_sync(FULL_MASK, dg);
            const int base = dg < GR_BINS ? whist[w][dg] : 0;
            rank[r] = base + __popc(peers & lanemask_lt());
            __syncwarp();
            if (dg < GR_BINS && (peers & lanemask_lt()) == 0u)
                whist[w][dg] = (unsigned short)(base + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        // the warps' counts to starts within the tile; run[]: the tile's counts of this thread's digits
        int run[PER];
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int b = tid + q * GR_THREADS;
            run[q] = 0;
            if (b < bins)
                for (int z = 0; z < GR_WARPS; z++) {
                    const int c = whist[z][b];
                    whist[z][b] = (unsigned short)run[q];
                    run[q] += c;
                }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < GR_ITEMS; r++) {
            if (key[r] >= 0) {
                const int dg = (key[r] >> shift) & (bins - 1);
                const int pos = start[dg] + whist[w][dg] + rank[r];
                if (keys_out)
                    keys_out[pos] = key[r];
                vals_out[pos] = val[r];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PER; q++)
            if (tid + q * GR_THREADS < bins)
                start[tid + q * GR_THREADS] += run[q];
    }
}

// offsets[r] = the number of sorted keys below r (r <= k), counts[r] = offsets[r + 1] - offsets[r].
__global__ void __launch_bounds__(GR_THREADS) k_group_offsets(const int32_t *__restrict__ keys, int64_t n, int32_t k,
                                                              int32_t *__restrict__ offsets,
                                                              int32_t *__restrict__ counts)
{
    const int64_t r = (int64_t)blockIdx.x * GR_THREADS + threadIdx.x;
    auto below = [&](int64_t v) {
        int64_t lo = 0, hi = n;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (keys[mid] < v)
                lo = mid + 1;
            else
                hi = mid;
        }
        return (int32_t)lo;
    };
    const int32_t a = r <= k ? below(r) : 0;
    int32_t b = __shfl_down_sync(FULL_MASK, a, 1);
    if (r > k)
        return;
    offsets[r] = a;
    if (counts && r < k) {
        if (lane_id() == 31)
            b = below(r + 1);
        counts[r] = b - a;
    }
}

// Passes over the bits of every sort key 0..k (k: the key of an out-of-range label), and bits per pass.
static int radix_passes(int32_t k, int *bits)
{
    uint32_t top = (uint32_t)k;
    int all = 0;
    while (top) {
        all++;
        top >>= 1;
    }
    const int passes = (all + GR_BITS - 1) / GR_BITS;  // at least one (k >= 1)
    *bits = (all + passes - 1) / passes;
    return passes;
}

static int radix_blocks(int64_t n)
{
    const int64_t tiles = (n + GR_TILE - 1) / GR_TILE;
    return (int)(tiles < GR_BLOCKS ? tiles : GR_BLOCKS);
}

size_t group_scratch_bytes(int64_t n, int32_t)
{
    size_t b = 0;
    auto add = [&](size_t bytes) { b += (bytes + 255) & ~size_t(255); };
    for (int q = 0; q < 4; q++)
        add(sizeof(int32_t) * (size_t)n);  // keys / values, two buffers each, aligned one by one
    add(sizeof(int32_t) * (size_t)GR_BINS * (size_t)radix_blocks(n));
    add(sizeof(int32_t) * GR_BINS);
    return b;
}

cudaError_t launch_group(const int32_t *labels, int64_t n, int32_t k, int32_t *offsets, int32_t *members,
                         int32_t *counts_out, void *scratch, DevStatus *st, cudaStream_t s, unsigned *zero)
{
    const int nblocks = radix_blocks(n);
    Carver cv{static_cast<char *>(scratch), 0, 0};
    int32_t *kbuf0 = cv.take<int32_t>((size_t)n);
    int32_t *kbuf1 = cv.take<int32_t>((size_t)n);
    int32_t *vbuf0 = cv.take<int32_t>((size_t)n);
    int32_t *vbuf1 = cv.take<int32_t>((size_t)n);
    int32_t *hist = cv.take<int32_t>((size_t)GR_BINS * (size_t)nblocks);
    int32_t *total = cv.take<int32_t>(GR_BINS);
    const int64_t tiles = (n + GR_TILE - 1) / GR_TILE, per = (tiles + nblocks - 1) / nblocks;
    int bits;
    const int passes = radix_passes(k, &bits), bins = 1 << bits;
    const int32_t *kin = labels;
    const int32_t *vin = nullptr;
    for (int p = 0; p < passes; p++) {
        const bool last = p == passes - 1;
        int32_t *kout = passes == 1 ? nullptr : (p & 1 ? kbuf1 : kbuf0);
        int32_t *vout = last ? members : (p & 1 ? vbuf1 : vbuf0);
        const int shift = p * bits;
        k_radix_hist<<<nblocks, GR_THREADS, 0, s>>>(kin, n, k, shift, bins, per, hist, p == 0 ? st : nullptr,
                                                    p == 0 ? zero : nullptr);
        k_radix_cols<<<(bins + GR_WARPS - 1) / GR_WARPS, GR_THREADS, 0, s>>>(hist, nblocks, bins, total);
        k_radix_scatter<<<nblocks, GR_THREADS, 0, s>>>(kin, vin, n, k, shift, bins, per, hist, total, kout, vout,
                                                       passes == 1 ? offsets : nullptr, counts_out);
        kin = kout;
        vin = vout;
    }
    if (passes > 1)
        k_group_offsets<<<(unsigned)(((int64_t)k + 1 + GR_THREADS - 1) / GR_THREADS), GR_THREADS, 0, s>>>(kin, n, k, offsets,
                                                                                                 counts_out);
    return cudaGetLastError();
}

}  // namespace gkm
