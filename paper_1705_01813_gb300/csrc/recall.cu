// Top-1 recall of a KNN graph, estimated on sampled queries (Sec. 5: the
// recall of the top-1 neighbour, taken over randomly chosen samples where the
// full ground truth is too costly).  For each query q its exact nearest
// neighbour is found by brute force over all n samples, pair distances in the
// canonical FP32 order (tiles.cuh) and ties by the smaller id (the graph's key
// order); the query is a hit when that neighbour is the first entry of q's
// graph row.  With exact distances in rows sorted by key, the true neighbour
// is in a row exactly when it is its first entry, so this is also the
// fraction of queries whose row holds their nearest neighbour.
//
// k_nn_tiles: block (b, s) takes the 64 queries of query block b and the
// samples of slice s, 64 at a time, as 64 x 64 distance tiles; each warp keeps
// the smallest (distance, id) key of eight queries over the slice, and the
// slices meet in best[] by atomic minimum.  Where there is enough to screen
// (recall_screened) the tensor cores find the keys first (recall_tc.cu) and
// the tiles take only the queries that are left, mostly none.
// k_nn_finish: the hit test, and the count of hits.
#include "common.cuh"
#include "merge.cuh"
#include "recall.cuh"
#include "tiles.cuh"

#include <cuda_bf16.h>

#include <type_traits>

namespace gkm {

constexpr int NN_T = 64;                                       // queries and samples per tile
constexpr size_t NN_SMEM = RefineTile<NN_T>::fixed_bytes + sizeof(uint64_t) * NN_T;

static int64_t nn_qblocks(int32_t m) { return ((int64_t)m + NN_T - 1) / NN_T; }

// slices of the samples per query block: about three blocks per SM in all
int recall_slices(int64_t n, int32_t m)
{
    const int64_t tiles = (n + NN_T - 1) / NN_T;
    int64_t s = (152 * 3 + nn_qblocks(m) - 1) / nn_qblocks(m);
    s = s < 1 ? 1 : s;
    return (int)(s > tiles ? tiles : s);
}

// The screening pays from RECALL_SCREEN_MIN pair coordinates on: 10,000 x 128, 1,000 queries 144 against 184 us,
// 1M x 32, 40 queries 203 against 243, 8,000 x 960, 200 queries 221 against 250; at 6.4e8 (10,000 x 64, 1,000 queries)
// the tiles take 110 us, the screening's seven launches and 256 queries at a time about as much.
constexpr double RECALL_SCREEN_MIN = 1.0e9;
// Nor does it for rows of fewer values: BF16's rounding is then as large as the distances to thousands of samples, and
// the lists overflow.  FP32 tiles against screening, us, graph rows with the true neighbour: Gaussian 400k x 2, 1,300
// queries 1,769 / 3,153, 1M x 1, 1,000 queries 3,425 / 5,081, 4M x 3, 300 queries 4,608 / 5,263; 400k x 4, 1,000 queries
// 1,495 / 435.  (Wider rows whose norm lies in one column lose as well: 400k x 32 2,216 / 3,006, 400k x 128, 500 queries
// 2,657 / 3,435, 1M x 128 16,154 / 14,802.)
constexpr int64_t RECALL_SCREEN_MIN_D = 4;

static bool recall_screened(int64_t n, int64_t d, int32_t m)
{
    return d >= RECALL_SCREEN_MIN_D && (double)n * (double)d * (double)m >= RECALL_SCREEN_MIN;
}

static size_t best_bytes(int32_t m) { return ((size_t)m * sizeof(uint64_t) + 255) & ~size_t(255); }

size_t recall_scratch_bytes(int64_t n, int64_t d, int32_t m)
{
    return best_bytes(m) + (recall_screened(n, d, m) ? recall_screen_bytes(d, m) : 0);
}

template <typename XT>
__global__ void __launch_bounds__(RF_THREADS) k_nn_tiles(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                        const int32_t *__restrict__ queries, int m, int slices,
                                                        const int32_t *__restrict__ left,
                                                        const int32_t *__restrict__ nleft,
                                                        uint64_t *__restrict__ bestq,
                                                        unsigned long long *__restrict__ hits, DevStatus *st)
{
    using TL = RefineTile<NN_T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *xr = reinterpret_cast<float *>(smem_raw);  // staging buffers of the pair tiles (tiles.cuh)
    float *dt = xr;  // aliases the staging buffers
    constexpr size_t span = TL::stage_floats > TL::tile_floats ? TL::stage_floats : TL::tile_floats;
    int *rid = reinterpret_cast<int *>(xr + span);
    int *cid = rid + NN_T;
    uint64_t *best = reinterpret_cast<uint64_t *>(cid + NN_T);
    const int tid = threadIdx.x, w = tid >> 5, lane = lane_id();
    if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0)
        *hits = 0ull;  // k_nn_finish counts; a clear of its own was a launch more (5,000 x 24, 100 queries 34 us, 32 so)
    // left (may be NULL): the queries to take, *nleft of them, instead of all m
    const int q0 = blockIdx.x * NN_T, nr = min(NN_T, (left ? *nleft : m) - q0);
    if (nr <= 0)
        return;
    auto index = [&](int t) { return left ? left[q0 + t] : q0 + t; };
    const int64_t tiles = (n + NN_T - 1) / NN_T;
    const int64_t t_lo = tiles * blockIdx.y / slices, t_hi = tiles * (blockIdx.y + 1) / slices;
    if (tid < NN_T) {
        int q = tid < nr ? queries[index(tid)] : -1;
        if (q >= n) {
            flag_error(st, GK_ERR_INVALID, (unsigned)index(tid));
            q = -1;
        }
        rid[tid] = q;
        best[tid] = ~0ull;
    }
    for (int64_t t = t_lo; t < t_hi; t++) {
        const int64_t j0 = t * NN_T;
        __syncthreads();  // the previous tile's distances are read
        if (tid < NN_T)
            cid[tid] = j0 + tid < n ? (int)(j0 + tid) : -1;
        __syncthreads();
        tile_distances<NN_T, false, false>(X, d, ld, rid, cid, tid >> 4, tid & 15,
                                           RefineTile<NN_T>::Q * (tid >> 4) < nr, xr, dt);
        __syncthreads();
        // warp w: queries w, w + 8, ..., the smallest key of the tile's samples other than the query
        for (int row = w; row < nr; row += RF_WARPS) {
            const int q = rid[row];
            uint64_t kmin = ~0ull;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int c = lane + 32 * h, j = cid[c];
                if (j >= 0 && j != q)
                    kmin = min(kmin, pack_key(dt[row * TL::DS + c], j));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                kmin = min(kmin, (uint64_t)__shfl_xor_sync(FULL_MASK, (unsigned long long)kmin, o));
            if (lane == 0 && kmin < best[row])
                best[row] = kmin;
        }
    }
    __syncthreads();
    if (tid < nr)
        atomicMin(reinterpret_cast<unsigned long long *>(bestq + index(tid)), (unsigned long long)best[tid]);
}

__global__ void k_nn_finish(const uint64_t *__restrict__ best, int m, const int32_t *__restrict__ queries, int64_t n,
                            const int32_t *__restrict__ g_idx, int kappa, int32_t *__restrict__ nn_idx,
                            float *__restrict__ nn_dist, unsigned long long *__restrict__ hits)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= m)
        return;
    const uint64_t k = best[q];
    const int qi = queries[q];
    const bool found = k != ~0ull && qi >= 0 && qi < n;
    const int id = found ? key_id(k) : -1;
    if (nn_idx)
        nn_idx[q] = id;
    if (nn_dist)
        nn_dist[q] = found ? key_dist(k) : __int_as_float(0x7f800000);
    if (found && __ldg(g_idx + (int64_t)qi * kappa) == id)
        atomicAdd(hits, 1ull);
}

template <typename XT>
static cudaError_t recall_t(const XT *X, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx, int32_t kappa,
                            const int32_t *queries, int32_t m, int32_t *nn_idx, float *nn_dist, int64_t *hits,
                            void *scratch, DevStatus *st, cudaStream_t s)
{
    cudaError_t e = set_max_smem(reinterpret_cast<const void *>(k_nn_tiles<XT>), (int)NN_SMEM);
    if (e != cudaSuccess)
        return e;
    const int slices = recall_slices(n, m);
    auto *count = reinterpret_cast<unsigned long long *>(hits);
    uint64_t *best = static_cast<uint64_t *>(scratch);
    if ((e = cudaMemsetAsync(best, 0xff, sizeof(uint64_t) * (size_t)m, s)) != cudaSuccess)
        return e;
    const int32_t *left = nullptr, *nleft = nullptr;
    if (recall_screened(n, d, m) &&
        (e = launch_recall_screen(X, std::is_same_v<XT, __nv_bfloat16>, n, d, ld, g_idx, kappa, queries, m, best,
                                  static_cast<char *>(scratch) + best_bytes(m), &left, &nleft, st, s)) != cudaSuccess)
        return e;
    const dim3 grid((unsigned)nn_qblocks(m), (unsigned)slices);
    k_nn_tiles<XT><<<grid, RF_THREADS, NN_SMEM, s>>>(X, n, d, ld, queries, m, slices, left, nleft, best, count, st);
    k_nn_finish<<<(m + 255) / 256, 256, 0, s>>>(best, m, queries, n, g_idx, kappa, nn_idx, nn_dist, count);
    return cudaGetLastError();
}

cudaError_t launch_recall(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx,
                          int32_t kappa, const int32_t *queries, int32_t m, int32_t *nn_idx, float *nn_dist,
                          int64_t *hits, void *scratch, DevStatus *st, cudaStream_t s)
{
    if (bf16)
        return recall_t(static_cast<const __nv_bfloat16 *>(X), n, d, ld, g_idx, kappa, queries, m, nn_idx, nn_dist,
                        hits, scratch, st, s);
    return recall_t(static_cast<const float *>(X), n, d, ld, g_idx, kappa, queries, m, nn_idx, nn_dist, hits, scratch,
                    st, s);
}

}  // namespace gkm
