// Two-means tree (Alg. 1, Sec. 3.2): k clusters by repeated bisection of the
// largest cluster into two halves of equal size.
//
// Every bisection halves a cluster (half u takes ceil(m/2) members), so the
// sizes in the tree depend on n and k only: the clusters of depth L have
// floor(n / 2^L) or that plus one members, whole depths are split before the
// next depth starts (a child is never larger than a cluster left at its
// parent's depth, and the shallower cluster goes first among equal sizes), and
// when k is not a power of two the last depth splits its larger clusters
// first, leftmost first.  The kernels therefore run one depth at a time over
// all of its clusters at once.  A cluster is a range [off, off + m) of a
// permutation of the samples; the permutation keeps each cluster's members in
// ascending id, and cluster j of depth L has the range that the bits of j
// (most significant first, 0 = u) pick out from the root.
//
// One bisection (each step over every cluster of the depth):
//   seeds    the two members with the smallest (draw(seed ^ TREE, L * 2^32 + id), id)
//   iters x  Lloyd 2-means: a member joins u when d(x, c_u) <= d(x, c_v), then
//            each centre becomes the FP32 rounding of the FP64 mean of its half
//            (an empty half keeps its centre)
//   keys     (d(x, c_u) - d(x, c_v) in FP32, id) as one ordered 64-bit word
//   select   the ceil(m/2)-th smallest key of the cluster (radix select)
//   split    members with a key up to it form u, the rest v, each in the
//            order they had (a stable partition: ascending id again)
// Distances are FP32 with one accumulator over ascending coordinates and one
// fused multiply-add per step, the decisions' precision.  Clusters are
// numbered left to right at the end.
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace gkm {
namespace {

constexpr uint64_t TAG_TREE = 0x5452454500000000ull;  // "TREE"
constexpr int TR_THREADS = 128;                       // pass kernel: one member per thread at a time
constexpr int TR_STAGE = 64;                          // coordinates staged per round
// Pitch of a staged row in elements (16 bytes more than its values): reads of four values of neighbouring rows, and of
// one value along a row, hit distinct banks (two-way for BF16's four).
template <typename XT>
constexpr int TR_VP = TR_STAGE + 16 / (int)sizeof(XT);
constexpr int64_t TR_CHUNK = 512;                     // members per chunk block; larger clusters take several
constexpr int SEL_THREADS = 256;
static_assert(TR_THREADS == 2 * TR_STAGE, "the sums give each coordinate two threads");

// Range of cluster j of depth L: the bits of j from the most significant, 0 = u (the left ceil(m/2)).
__device__ __forceinline__ void seg_geom(int64_t n, int L, int64_t j, int64_t &off, int64_t &m)
{
    off = 0;
    m = n;
    for (int b = L - 1; b >= 0; b--) {
        const int64_t h = (m + 1) >> 1;
        if ((j >> b) & 1) {
            off += h;
            m -= h;
        } else {
            m = h;
        }
    }
}

// Order-preserving map of an FP32 value to an unsigned word.
__device__ __forceinline__ uint32_t f32_order(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ bool hk_less(uint64_t ha, int ia, uint64_t hb, int ib)
{
    return ha < hb || (ha == hb && ia < ib);
}

// (h1, i1) <= (h2, i2) are the two smallest keys seen; merge another such pair (g1, j1) <= (g2, j2).
__device__ __forceinline__ void top2_merge(uint64_t &h1, int &i1, uint64_t &h2, int &i2, uint64_t g1, int j1,
                                           uint64_t g2, int j2)
{
    if (hk_less(g1, j1, h1, i1)) {  // the other pair's first wins; the second is the smaller of h1 and g2
        if (hk_less(h1, i1, g2, j2)) {
            h2 = h1;
            i2 = i1;
        } else {
            h2 = g2;
            i2 = j2;
        }
        h1 = g1;
        i1 = j1;
    } else if (hk_less(g1, j1, h2, i2)) {
        h2 = g1;
        i2 = j1;
    }
}

// Radix selection step, one full warp: over a 256-bin histogram, the digit whose cumulative count first exceeds
// rank and the number of keys below that digit (lane q reads bins 8q .. 8q + 7).  The caller guarantees that
// the bins hold more than rank keys.
__device__ __forceinline__ void warp_pick(const unsigned *hist, int64_t rank, int &digit, int64_t &below)
{
    const int lane = threadIdx.x & 31;
    unsigned own = 0;
    for (int q = 0; q < 8; q++)
        own += hist[8 * lane + q];
    unsigned incl = own;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o)
            incl += v;
    }
    const unsigned hit = __ballot_sync(FULL_MASK, (int64_t)incl > rank);
    const int first = hit ? __ffs(hit) - 1 : 31;
    int dg = 8 * lane + 7;
    int64_t base = 0;
    if (lane == first) {
        base = incl - own;
        for (int q = 0; q < 8; q++) {
            const unsigned h = hist[8 * lane + q];
            if (base + (int64_t)h > rank) {
                dg = 8 * lane + q;
                break;
            }
            base += h;
        }
    }
    digit = __shfl_sync(FULL_MASK, dg, first);
    below = __shfl_sync(FULL_MASK, base, first);
}

__global__ void k_tree_iota(int32_t *perm, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        perm[i] = (int32_t)i;
}

// Last, partial depth L: which of its S = 2^L clusters split (r of them, the larger first, then the leftmost) and
// how many split before each.  One block.
__global__ void __launch_bounds__(1024) k_tree_plan(int64_t n, int L, int64_t r, int32_t *spl, int32_t *pre)
{
    __shared__ int wsum[32];
    const int64_t S = (int64_t)1 << L;
    const int64_t a = n >> L;
    const int64_t r1 = min(r, n - a * S);  // larger clusters (a + 1 members) split
    const int64_t r0 = r - r1;             // clusters of a members split
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t carry = 0;
    for (int64_t t0 = 0; t0 < S; t0 += blockDim.x) {
        const int64_t j = t0 + threadIdx.x;
        bool big = false;
        if (j < S) {
            int64_t off, m;
            seg_geom(n, L, j, off, m);
            big = m == a + 1;
        }
        const unsigned bal = __ballot_sync(FULL_MASK, big);
        if (lane == 0)
            wsum[warp] = __popc(bal);
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            before += w < warp ? wsum[w] : 0;
            total += wsum[w];
        }
        const int64_t rank1 = carry + before + __popc(bal & lanemask_lt());
        if (j < S) {
            const int64_t rank0 = j - rank1;
            spl[j] = big ? (rank1 < r1) : (rank0 < r0);
            pre[j] = (int32_t)(min(rank1, r1) + min(rank0, r0));
        }
        carry += total;
        __syncthreads();
    }
}

// Chunk c of cluster j: C chunks of nearly equal length over the cluster's range.
__device__ __forceinline__ void chunk_range(int64_t off, int64_t m, int64_t C, int64_t c, int64_t &b, int64_t &e)
{
    b = off + c * m / C;
    e = off + (c + 1) * m / C;
}

struct Top2 {
    uint64_t h1, h2;
    int32_t i1, i2;
};

// Seeds, first step: the two members of smallest (draw, id) in every chunk of a splitting cluster.
__global__ void __launch_bounds__(SEL_THREADS) k_tree_seed_part(int64_t n, int L, int64_t C,
                                                                 const int32_t *__restrict__ perm,
                                                                 const int32_t *__restrict__ spl, uint64_t seed,
                                                                 Top2 *__restrict__ part)
{
    __shared__ Top2 sw[SEL_THREADS / 32];
    const int64_t j = blockIdx.x / C, c = blockIdx.x % C;
    if (spl && !spl[j])
        return;
    int64_t off, m, b, e;
    seg_geom(n, L, j, off, m);
    chunk_range(off, m, C, c, b, e);
    const uint64_t key = seed ^ TAG_TREE;
    uint64_t h1 = ~0ull, h2 = ~0ull;
    int i1 = INT32_MAX, i2 = INT32_MAX;
    for (int64_t p = b + threadIdx.x; p < e; p += SEL_THREADS) {
        const int id = perm[p];
        top2_merge(h1, i1, h2, i2, sm64_draw(key, ((uint64_t)(uint32_t)L << 32) | (uint32_t)id), id, ~0ull,
                   INT32_MAX);
    }
    for (int o = 16; o > 0; o >>= 1)
        top2_merge(h1, i1, h2, i2, __shfl_xor_sync(FULL_MASK, h1, o), __shfl_xor_sync(FULL_MASK, i1, o),
                   __shfl_xor_sync(FULL_MASK, h2, o), __shfl_xor_sync(FULL_MASK, i2, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        sw[warp] = Top2{h1, h2, i1, i2};
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < SEL_THREADS / 32; w++)
            top2_merge(h1, i1, h2, i2, sw[w].h1, sw[w].i1, sw[w].h2, sw[w].i2);
        part[blockIdx.x] = Top2{h1, h2, i1, i2};
    }
}

// Seeds, second step: merge the chunks' pairs; the two winners' rows become the starting centres c_u, c_v
// (cen: 2 x d floats per cluster).
template <typename XT>
__global__ void __launch_bounds__(TR_THREADS) k_tree_seed_final(const XT *__restrict__ X, int64_t n, int d,
                                                                 int64_t ld, int64_t C,
                                                                 const int32_t *__restrict__ spl,
                                                                 const Top2 *__restrict__ part,
                                                                 float *__restrict__ cen, DevStatus *st)
{
    __shared__ int s_id[2];
    const int64_t j = blockIdx.x;
    if (spl && !spl[j])
        return;
    if (threadIdx.x < 32) {
        uint64_t h1 = ~0ull, h2 = ~0ull;
        int i1 = INT32_MAX, i2 = INT32_MAX;
        for (int64_t c = threadIdx.x; c < C; c += 32) {
            const Top2 t = part[j * C + c];
            top2_merge(h1, i1, h2, i2, t.h1, t.i1, t.h2, t.i2);
        }
        for (int o = 16; o > 0; o >>= 1)
            top2_merge(h1, i1, h2, i2, __shfl_xor_sync(FULL_MASK, h1, o), __shfl_xor_sync(FULL_MASK, i1, o),
                       __shfl_xor_sync(FULL_MASK, h2, o), __shfl_xor_sync(FULL_MASK, i2, o));
        if (threadIdx.x == 0) {
            if ((unsigned)i1 >= (unsigned)n || (unsigned)i2 >= (unsigned)n) {
                flag_error(st, GK_ERR_INVALID, (unsigned)j);
                i1 = i2 = 0;
            }
            s_id[0] = i1;
            s_id[1] = i2;
        }
    }
    __syncthreads();
    const XT *xa = X + (int64_t)s_id[0] * ld, *xb = X + (int64_t)s_id[1] * ld;
    float *cj = cen + j * 2 * (int64_t)d;
    for (int t = threadIdx.x; t < d; t += TR_THREADS) {
        cj[t] = ldx(xa + t);
        cj[d + t] = ldx(xb + t);
    }
}

// Largest magnitude of every column, as the bits of its float (infinities and NaN above every number): colmax[d], zeroed.
template <typename XT>
__global__ void __launch_bounds__(256) k_tree_colmax(const XT *__restrict__ X, int64_t n, int d, int64_t ld, bool vec,
                                                     unsigned *__restrict__ colmax)
{
    __shared__ unsigned s_mx[128];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, col = blockIdx.y * 128 + lane * 4;
    if (threadIdx.x < 128)
        s_mx[threadIdx.x] = 0u;
    __syncthreads();
    unsigned mx[4] = {0u, 0u, 0u, 0u};
    if (col < d) {
#pragma unroll 4
        for (int64_t i = (int64_t)blockIdx.x * 8 + warp; i < n; i += (int64_t)gridDim.x * 8) {
            const XT *p = X + i * ld + col;
            if (vec) {
                const float4 v = ldx4<XT>(p);
                mx[0] = max(mx[0], __float_as_uint(fabsf(v.x)));
                mx[1] = max(mx[1], __float_as_uint(fabsf(v.y)));
                mx[2] = max(mx[2], __float_as_uint(fabsf(v.z)));
                mx[3] = max(mx[3], __float_as_uint(fabsf(v.w)));
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (col + q < d)
                        mx[q] = max(mx[q], __float_as_uint(fabsf(ldx(p + q))));
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; q++)
        atomicMax(&s_mx[lane * 4 + q], mx[q]);
    __syncthreads();
    const int t = blockIdx.y * 128 + threadIdx.x;
    if (threadIdx.x < 128 && t < d)
        atomicMax(colmax + t, s_mx[threadIdx.x]);
}

// ---------------------------------------------------------------------------
// The centres.  A centre is defined as the FP32 rounding of an FP64 mean whose sum runs over the members in ascending id
// (chunk by chunk, the chunks' sums in order), and the FP64 pipe would bound the tree: one addition per member and
// coordinate, 0.5 a cycle and SM, was 70% of it.  The sums are taken in integers instead, which no order changes.  With
// column t's largest magnitude below 2^(e + 1), y = x 2^(20 - e) is below 2^21 and split exactly as
//   y = h0 + h1 2^-22 + h2 2^-44 + error,  |error| <= 2^-45,
// h0, h1, h2 integers of at most 2^21 (the sum of y 2^22 and 1.5 2^23 rounds to an integer in the float's low bits).
// Where every h1 is zero, or every h2 and at most 1024 members are summed (and y itself is exact: no scaling down),
// all partial sums are multiples of one unit that FP64 holds exactly, so the ordered FP64 sum is this sum.  Otherwise
// the two means differ by at most (chunk + chunks) 2^-53 mean|x| plus the split's remainder, and their FP32 roundings
// are the same unless the mean lies that close to the midpoint of two floats: a few centre coordinates in 10^6, more
// where a mean is small beside its members.  Those get the code REDO and k_tree_redo sums them in the defined order.
// So every centre has the bits of the definition.
// ---------------------------------------------------------------------------
constexpr unsigned REDO = 0x7fb0dead;  // a NaN no mean takes
constexpr float SPLIT_M = 12582912.f;  // 1.5 2^23
constexpr int REDO_CAP = 1 << 16;      // listed coordinates, at most

// The coordinates coded REDO in the current pass: their number, which may exceed the list's room (cap entries).
struct RedoList {
    unsigned *n;
    int64_t *at;
    int cap;
};

// Writes a centre coordinate and lists it when it is to be summed again.
__device__ __forceinline__ void put_centre(float *cen, int64_t z, unsigned bits, const RedoList &redo)
{
    cen[z] = __uint_as_float(bits);
    if (bits == REDO) {
        const unsigned i = atomicAdd(redo.n, 1u);
        if (i < (unsigned)redo.cap)
            redo.at[i] = z;
    }
}

// 2^(20 - e) for a column whose largest magnitude has the given bits; 0 when it is not finite.
__device__ __forceinline__ float col_scale(unsigned mx)
{
    const int e = max((int)(mx >> 23) - 127, -106);  // 2^126 at most
    return mx >= 0x7f800000u ? 0.f : __uint_as_float((unsigned)(20 - e + 127) << 23);
}

// The centre coordinate of cnt > 0 members from their limb sums, or REDO.  any: bit 0 a second limb, bit 1 a third limb
// or remainder occurred; mass: the sum of |y|, added in any order.
__device__ __forceinline__ unsigned centre_bits(int64_t h0, int64_t h1, int64_t h2, unsigned any, float mass,
                                                int64_t cnt, unsigned mx, int64_t chunks)
{
    const float sc = col_scale(mx);
    if (sc == 0.f)
        return REDO;
    const double y = (double)h0 + ((double)h1 * 0x1p-22 + (double)h2 * 0x1p-44);
    const double q = y / (double)sc / (double)cnt;  // the scaling is exact
    const unsigned f = __float_as_uint((float)q);
    if (sc >= 1.f && (any == 0 || (any == 1 && cnt <= 1024)))
        return f;
    const uint64_t bits = (uint64_t)__double_as_longlong(q);
    const int e = (int)((bits >> 52) & 0x7ff) - 1023;
    if (e < -126 || e >= 127)  // outside FP32's normal range, or zero
        return REDO;
    // distance of q from the midpoint of its two floats, and the bound, in units of q's last place, 2^(e - 52)
    const int64_t frac = (int64_t)(bits & 0x1fffffffull) - 0x10000000ll;
    const double rel = ((double)(TR_CHUNK + 8) + (double)chunks) * (1.02 + (double)chunks * 0x1p-23) * 0x1p-53;
    const double tol = ((double)mass * rel / (double)cnt + 0x1p-44) / (double)sc;
    const double units = tol * __longlong_as_double((long long)(52 - e + 1023) << 52) + 4.0;
    return (double)llabs(frac) <= units ? REDO : f;
}

// Dynamic shared memory of the pass kernel: limb sums, masses and flags of both halves, both centres, the staged rows,
// the block's member ids and counts, the rows by half.
template <typename XT>
__host__ __device__ constexpr size_t pass_smem(int d)
{
    return (size_t)44 * d + sizeof(XT) * TR_THREADS * TR_VP<XT> + 2 * sizeof(int) * TR_THREADS + TR_THREADS + 64;
}

// Four staged values, widened exactly.
__device__ __forceinline__ float4 staged4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 staged4(const __nv_bfloat16 *p)
{
    return bf16x4_to_float4(*reinterpret_cast<const uint2 *>(p));
}

// One pass over the members of every splitting cluster of depth L, C chunks per cluster (grid S x C).  Each thread
// takes one member at a time: the rows of the block's 128 members are staged 64 coordinates at a time and each
// thread sums its member's two distances in the canonical FP32 order (both at once in packed FP32x2).
//   KEYS = false (a Lloyd iteration): the member joins u when d_u <= d_v and its row is added to its half's limb sums
//     (the stages again, the last one first as it is still there; threads share out coordinates and rows); with one chunk
//     the block writes the new centres, otherwise its sums and counts are added to acc, mass, flg and cnts, for
//     k_tree_centres.  halves[p] is the half, for k_tree_redo.
//   KEYS = true: keys[p] = (order(d_u - d_v) << 32) | id.
// Bound by the reads of the rows: 1M x 128 FP32 (512 MB) takes 84 us with KEYS, 6.1 TB/s, and 159 us without (all but
// the last stage are read again, mostly from the L2, and the sums).  With loads through registers, four in flight, it
// was 229 and 332 us (BF16 225 and 337, now 64 and 150); before the packed distances and the integer sums 421 and 879
// us, the FP64 additions' time.  Two stage buffers, the next stage in flight during the distances, leave 3 blocks of an
// SM instead of 5: 91 and 174 us.
template <typename XT, bool KEYS>
__global__ void __launch_bounds__(TR_THREADS) k_tree_pass(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                          bool vec, int L, int64_t C, const int32_t *__restrict__ perm,
                                                          const int32_t *__restrict__ spl, float *__restrict__ cen,
                                                          const unsigned *__restrict__ colmax,
                                                          unsigned long long *__restrict__ acc,
                                                          unsigned *__restrict__ flg, float *__restrict__ mass,
                                                          unsigned *__restrict__ cnts, uint8_t *__restrict__ halves,
                                                          uint64_t *__restrict__ keys, const RedoList redo, DevStatus *st)
{
    extern __shared__ __align__(16) unsigned char tr_smem[];
    constexpr int VP = TR_VP<XT>;
    XT *stage = reinterpret_cast<XT *>(tr_smem);                       // [TR_THREADS][TR_VP]
    int *sid = reinterpret_cast<int *>(stage + TR_THREADS * VP);
    int *s_n = sid + TR_THREADS;                                             // members of u, of u and v in the group
    unsigned char *order = reinterpret_cast<unsigned char *>(s_n + TR_THREADS);  // rows of u, then of v
    float2 *cuv = reinterpret_cast<float2 *>(order + TR_THREADS);            // [d]: (c_u, c_v)
    int *lsum = reinterpret_cast<int *>(cuv + d);                            // [2][3][d]
    float *lmass = reinterpret_cast<float *>(lsum + 6 * (size_t)d);          // [2][d]
    unsigned *lany = reinterpret_cast<unsigned *>(lmass + 2 * (size_t)d);    // [d], two bits per half
    const int64_t j = blockIdx.x / C, c = blockIdx.x % C;
    if (spl && !spl[j])
        return;
    int64_t off, m, b, e;
    seg_geom(n, L, j, off, m);
    chunk_range(off, m, C, c, b, e);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *cj = cen + j * 2 * (int64_t)d;
    for (int t = tid; t < d; t += TR_THREADS)
        cuv[t] = make_float2(cj[t], cj[d + t]);
    if (!KEYS)
        for (int t = tid; t < 9 * d; t += TR_THREADS)  // the masses and flags too
            lsum[t] = 0;
    const int nst = (d + TR_STAGE - 1) / TR_STAGE;
    // the 64 coordinates of stage s of the block's gn rows (zeros past d), all in flight at once: 16 lanes per row, or a
    // lane per coordinate
    int gn = 0;
    auto stage_rows = [&](int s) {
        const int t0 = s * TR_STAGE;
        if (vec) {
            const int t = t0 + (tid & 15) * 4;
            XT *to = stage + (tid & 15) * 4;
#pragma unroll 8
            for (int r = tid >> 4; r < gn; r += TR_THREADS / 16) {
                XT *q = to + r * VP;
                const XT *x = X + (int64_t)sid[r] * ld + t;
                if constexpr (std::is_same_v<XT, float>) {
                    if (t < d)
                        cp_async16(q, x);
                    else
                        *reinterpret_cast<uint4 *>(q) = make_uint4(0u, 0u, 0u, 0u);
                } else {
                    if (t < d)
                        cp_async8(q, x);
                    else
                        *reinterpret_cast<uint2 *>(q) = make_uint2(0u, 0u);
                }
            }
        } else {
            for (int r = warp; r < gn; r += TR_THREADS / 32)
                for (int q = lane; q < TR_STAGE; q += 32)
                    stage[r * VP + q] = t0 + q < d ? X[(int64_t)sid[r] * ld + t0 + q] : XT(0.f);
        }
        cp_async_wait_all();
    };
    __syncthreads();
    int64_t cnt_u = 0, cnt_v = 0;
    for (int64_t g = b; g < e; g += TR_THREADS) {
        const int64_t p = g + tid;
        const bool valid = p < e;
        gn = (int)min((int64_t)TR_THREADS, e - g);
        int id = perm[valid ? p : b];
        if ((unsigned)id >= (unsigned)n) {
            flag_error(st, GK_ERR_INVALID, (unsigned)j);
            id = 0;
        }
        sid[tid] = id;
        float2 duv = make_float2(0.f, 0.f);
        const float2 m1 = make_float2(-1.f, -1.f);
        for (int s = 0; s < nst; s++) {
            __syncthreads();  // sid written; the previous stage consumed
            stage_rows(s);
            __syncthreads();
            if (!valid)
                continue;
            const XT *xs = stage + tid * VP;
            const float2 *cs = cuv + s * TR_STAGE;
            const int tw = min(TR_STAGE, d - s * TR_STAGE);
            auto add = [&](float x, float2 cc) {
                const float2 ee = __ffma2_rn(cc, m1, make_float2(x, x));  // x - c, rounded once
                duv = __ffma2_rn(ee, ee, duv);
            };
            int tt = 0;
#pragma unroll 4
            for (; tt + 4 <= tw; tt += 4) {
                const float4 x = staged4(xs + tt);
                const float4 a = *reinterpret_cast<const float4 *>(cs + tt);
                const float4 h = *reinterpret_cast<const float4 *>(cs + tt + 2);
                add(x.x, make_float2(a.x, a.y));
                add(x.y, make_float2(a.z, a.w));
                add(x.z, make_float2(h.x, h.y));
                add(x.w, make_float2(h.z, h.w));
            }
            for (; tt < tw; tt++)
                add((float)xs[tt], cs[tt]);
        }
        if (KEYS) {
            if (valid) {
                const float dk = __fsub_rn(duv.x, duv.y);
                if (!isfinite(dk))
                    flag_error(st, GK_ERR_NUMERIC, (unsigned)id);
                keys[p] = ((uint64_t)f32_order(dk) << 32) | (uint32_t)id;
            }
        } else {
            // the group's rows by half
            const int half = duv.x <= duv.y ? 0 : 1;
            if (valid)
                halves[p] = (uint8_t)half;
            const unsigned bu = __ballot_sync(FULL_MASK, valid && half == 0);
            const unsigned bv = __ballot_sync(FULL_MASK, valid && half == 1);
            if (lane == 0) {
                s_n[warp] = __popc(bu);
                s_n[4 + warp] = __popc(bv);
            }
            __syncthreads();
            int nu = 0, nv = 0, au = 0, av = 0;
            for (int w = 0; w < TR_THREADS / 32; w++) {
                au += w < warp ? s_n[w] : 0;
                av += w < warp ? s_n[4 + w] : 0;
                nu += s_n[w];
                nv += s_n[4 + w];
            }
            if (valid)
                order[half == 0 ? au + __popc(bu & lanemask_lt()) : nu + av + __popc(bv & lanemask_lt())] =
                    (unsigned char)tid;
            cnt_u += nu;
            cnt_v += nv;
            __syncthreads();
            const int cc = tid % TR_STAGE, gg = tid / TR_STAGE;  // coordinate of the stage, rows gg, gg + 2, ...
            for (int s = nst - 1; s >= 0; s--) {
                if (s < nst - 1) {
                    __syncthreads();  // the stage before is consumed
                    stage_rows(s);
                    __syncthreads();
                }
                const int t = s * TR_STAGE + cc;
                const float sc = t < d ? col_scale(colmax[t]) : 0.f;
                if (sc != 0.f) {
                    auto half_sum = [&](int lo, int hi, int h) {
                        int s0 = 0, s1 = 0, s2 = 0;
                        float ms = 0.f;
                        unsigned a1 = 0, a2 = 0;
                        constexpr int MB = 0x4b400000;  // the bits of SPLIT_M
#pragma unroll 4
                        for (int r = lo + gg; r < hi; r += 2) {
                            const float y = (float)stage[order[r] * VP + cc] * sc;
                            const float t0 = __fadd_rn(y, SPLIT_M), r0 = __fsub_rn(y, __fsub_rn(t0, SPLIT_M));
                            const float t1 = __fmaf_rn(r0, 4194304.f, SPLIT_M);
                            const float r1 = __fmaf_rn(__fsub_rn(t1, SPLIT_M), -0x1p-22f, r0);
                            const float t2 = __fmaf_rn(r1, 0x1p44f, SPLIT_M);
                            ms += fabsf(y);
                            s0 += __float_as_int(t0) - MB;
                            s1 += __float_as_int(t1) - MB;
                            s2 += __float_as_int(t2) - MB;
                            a1 |= __float_as_uint(r0) << 1;  // without the sign of a zero
                            a2 |= __float_as_uint(r1) << 1;
                        }
                        atomicAdd(&lsum[(3 * h) * d + t], s0);
                        atomicAdd(&lmass[h * d + t], ms);
                        if (a1) {
                            atomicAdd(&lsum[(3 * h + 1) * d + t], s1);
                            atomicAdd(&lsum[(3 * h + 2) * d + t], s2);
                            atomicOr(&lany[t], (a2 ? 3u : 1u) << (2 * h));
                        }
                    };
                    half_sum(0, nu, 0);
                    half_sum(nu, nu + nv, 1);
                }
            }
        }
        __syncthreads();  // sid and order are rewritten by the next group
    }
    if (KEYS)
        return;
    if (C == 1) {
        for (int t = tid; t < 2 * d; t += TR_THREADS) {
            const int h = t >= d ? 1 : 0, tc = t - h * d;
            const int64_t cnt = h ? cnt_v : cnt_u;
            if (cnt)
                put_centre(cen, j * 2 * (int64_t)d + t,
                           centre_bits(lsum[3 * h * d + tc], lsum[(3 * h + 1) * d + tc], lsum[(3 * h + 2) * d + tc],
                                       (lany[tc] >> (2 * h)) & 3u, lmass[t], cnt, colmax[tc], 1),
                           redo);
        }
    } else {
        for (int t = tid; t < 6 * d; t += TR_THREADS)
            if (lsum[t])
                atomicAdd(acc + j * 6 * (int64_t)d + t, (unsigned long long)(long long)lsum[t]);
        for (int t = tid; t < 2 * d; t += TR_THREADS) {
            const int h = t >= d ? 1 : 0;
            const unsigned any = (lany[t - h * d] >> (2 * h)) & 3u;
            atomicAdd(mass + j * 2 * (int64_t)d + t, lmass[t]);
            if (any)
                atomicOr(flg + j * 2 * (int64_t)d + t, any);
        }
        if (tid == 0) {
            atomicAdd(cnts + 2 * j, (unsigned)cnt_u);
            atomicAdd(cnts + 2 * j + 1, (unsigned)cnt_v);
        }
    }
}

// Centres of the clusters of several chunks from their limb sums; acc, mass and flg are left zeroed for the next
// pass; k_tree_redo, which follows, clears cnts.
__global__ void __launch_bounds__(256) k_tree_centres(int64_t S, int d, int64_t C, const int32_t *__restrict__ spl,
                                                      float *__restrict__ cen, const unsigned *__restrict__ colmax,
                                                      unsigned long long *__restrict__ acc, unsigned *__restrict__ flg,
                                                      float *__restrict__ mass, const unsigned *__restrict__ cnts,
                                                      const RedoList redo)
{
    for (int64_t q = blockIdx.x * (int64_t)256 + threadIdx.x; q < S * 2 * d; q += (int64_t)gridDim.x * 256) {
        const int64_t j = q / (2 * d);
        if (spl && !spl[j])
            continue;
        const int t = (int)(q - j * 2 * d), h = t >= d ? 1 : 0, tc = t - h * d;
        unsigned long long *a = acc + j * 6 * (int64_t)d + 3 * h * (int64_t)d + tc;
        const int64_t cnt = cnts[2 * j + h];
        if (cnt)
            put_centre(cen, q,
                       centre_bits((int64_t)a[0], (int64_t)a[d], (int64_t)a[2 * (int64_t)d], flg[q], mass[q], cnt,
                                   colmax[tc], C),
                       redo);
        a[0] = a[d] = a[2 * (int64_t)d] = 0ull;
        flg[q] = 0u;
        mass[q] = 0.f;
    }
}

// The centre coordinates coded REDO, in the defined order (chunk by chunk in ascending id, the chunks' sums added in
// order): a warp per listed coordinate and chunk, which loads 32 members at a time; with several chunks their sums go
// to part (cap C <= n doubles, the keys' place) and the last block to finish adds them up.  The last block also clears
// the list and cnts (of several chunks) for the next pass.  When the list overflowed, all coordinates are looked
// through instead, a warp per coordinate and a lane per chunk.  (That form for every coordinate took up to 32 ms for
// one of the root of 1M members: one warp; this one 0.1.)
template <typename XT>
__global__ void __launch_bounds__(256) k_tree_redo(const XT *__restrict__ X, int64_t n, int d, int64_t ld, int L,
                                                   int64_t S, int64_t C, const int32_t *__restrict__ perm,
                                                   const uint8_t *__restrict__ halves, float *__restrict__ cen,
                                                   unsigned *__restrict__ cnts, double *__restrict__ part,
                                                   const RedoList redo, unsigned *__restrict__ ticket)
{
    const int lane = threadIdx.x & 31;
    const int64_t total = S * 2 * d, step = (int64_t)gridDim.x * 256;
    const unsigned listed = *redo.n;
    const bool all = listed > (unsigned)redo.cap;
    auto member = [&](int64_t p, int tc) {
        const int id = perm[p];
        return ldx(X + ((unsigned)id < (unsigned)n ? (int64_t)id * ld : 0) + tc);
    };
    if (!all) {
        const int64_t items = (int64_t)listed * C;
        for (int64_t it = (blockIdx.x * (int64_t)256 + threadIdx.x) >> 5; it < items; it += step >> 5) {
            const int64_t z = redo.at[it / C], c = it % C, j = z / (2 * d);
            const int t = (int)(z - j * 2 * d), h = t >= d ? 1 : 0, tc = t - h * d;
            int64_t off, m, b, e;
            seg_geom(n, L, j, off, m);
            chunk_range(off, m, C, c, b, e);
            double sum = 0.0;
            int cnt = 0;
            float x = b + lane < e ? member(b + lane, tc) : 0.f;
            int hl = b + lane < e ? halves[b + lane] : 2;
            for (int64_t p = b; p < e; p += 32) {
                const float x0 = x;
                unsigned mine = __ballot_sync(FULL_MASK, hl == h);
                const int64_t q = p + 32 + lane;
                x = q < e ? member(q, tc) : 0.f;
                hl = q < e ? halves[q] : 2;
                cnt += __popc(mine);
                while (mine) {
                    sum = __dadd_rn(sum, widen(__shfl_sync(FULL_MASK, x0, __ffs(mine) - 1)));
                    mine &= mine - 1;
                }
            }
            if (lane == 0) {
                if (C == 1)
                    cen[z] = (float)(sum / (double)cnt);
                else
                    part[it] = sum;
            }
        }
    } else {
        for (int64_t q0 = blockIdx.x * (int64_t)256 + (threadIdx.x & ~31); q0 < total; q0 += step) {
            const int64_t q = q0 + lane;
            unsigned left = __ballot_sync(FULL_MASK, q < total && __float_as_uint(cen[q]) == REDO);
            while (left) {
                const int64_t z = q0 + __ffs(left) - 1;
                left &= left - 1;
                const int64_t j = z / (2 * d);
                const int t = (int)(z - j * 2 * d), h = t >= d ? 1 : 0, tc = t - h * d;
                int64_t off, m;
                seg_geom(n, L, j, off, m);
                double total_sum = 0.0;
                long long cnt = 0;
                for (int64_t c0 = 0; c0 < C; c0 += 32) {
                    double sum = 0.0;
                    int nc = 0;
                    if (c0 + lane < C) {
                        int64_t b, e;
                        chunk_range(off, m, C, c0 + lane, b, e);
#pragma unroll 8
                        for (int64_t p = b; p < e; p++) {
                            const float x = member(p, tc);
                            if (halves[p] == h) {
                                sum = __dadd_rn(sum, widen(x));
                                nc++;
                            }
                        }
                    }
                    for (int s = 0; s < 32 && c0 + s < C; s++) {
                        total_sum = __dadd_rn(total_sum, __shfl_sync(FULL_MASK, sum, s));
                        cnt += __shfl_sync(FULL_MASK, nc, s);
                    }
                }
                if (lane == 0)
                    cen[z] = (float)(total_sum / (double)cnt);
            }
        }
    }
    if (!last_block(ticket))
        return;
    if (C > 1) {
        if (!all)
            for (int64_t i = threadIdx.x; i < listed; i += 256) {
                const int64_t z = redo.at[i], j = z / (2 * d);
                double sum = 0.0;
#pragma unroll 8
                for (int64_t c = 0; c < C; c++)
                    sum = __dadd_rn(sum, __ldcg(part + i * C + c));
                cen[z] = (float)(sum / (double)cnts[2 * j + (z - j * 2 * d >= d ? 1 : 0)]);
            }
        __syncthreads();  // the counts are read
        for (int64_t q = threadIdx.x; q < 2 * S; q += 256)
            cnts[q] = 0u;
    }
    if (threadIdx.x == 0) {
        *redo.n = 0u;
        *ticket = 0u;
    }
}

// The ceil(m/2)-th smallest key of every splitting cluster (keys are distinct: they end in the member's id), by
// radix selection over 8-bit digits from the most significant.  Clusters of one chunk: one block each.
__global__ void __launch_bounds__(SEL_THREADS) k_tree_select(int64_t n, int L, const int32_t *__restrict__ spl,
                                                             const uint64_t *__restrict__ keys,
                                                             uint64_t *__restrict__ thr)
{
    __shared__ unsigned hist[256];
    __shared__ uint64_t s_prefix;
    __shared__ int64_t s_rank;
    const int64_t j = blockIdx.x;
    if (spl && !spl[j])
        return;
    int64_t off, m;
    seg_geom(n, L, j, off, m);
    const int tid = threadIdx.x;
    uint64_t prefix = 0, mask = 0;
    int64_t rank = (m + 1) / 2 - 1;  // among the keys that match the prefix so far
    for (int shift = 56; shift >= 0; shift -= 8) {
        hist[tid] = 0;  // SEL_THREADS == 256 bins
        __syncthreads();
        for (int64_t p = off + tid; p < off + m; p += SEL_THREADS) {
            const uint64_t k = keys[p];
            if ((k & mask) == prefix)
                atomicAdd(&hist[(k >> shift) & 255], 1u);
        }
        __syncthreads();
        if (tid < 32) {
            int dg;
            int64_t below;
            warp_pick(hist, rank, dg, below);
            if (tid == 0) {
                s_prefix = prefix | ((uint64_t)dg << shift);
                s_rank = rank - below;
            }
        }
        __syncthreads();
        prefix = s_prefix;
        rank = s_rank;
        mask |= (uint64_t)255 << shift;
    }
    if (tid == 0)
        thr[j] = prefix;
}

// The same selection for clusters of several chunks, one digit at a time: k_tree_sel_init, then per digit
// k_tree_hist (every chunk adds its histogram of the keys that match the prefix) and k_tree_digit (one warp per
// cluster picks the digit and clears the histogram).  thr holds the prefix, srank the rank within it.
__global__ void __launch_bounds__(SEL_THREADS) k_tree_sel_init(int64_t n, int L, const int32_t *__restrict__ spl,
                                                               uint64_t *__restrict__ thr, int64_t *__restrict__ srank,
                                                               unsigned *__restrict__ ghist)
{
    const int64_t j = blockIdx.x;
    if (spl && !spl[j])
        return;
    int64_t off, m;
    seg_geom(n, L, j, off, m);
    ghist[j * 256 + threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        thr[j] = 0;
        srank[j] = (m + 1) / 2 - 1;
    }
}

__global__ void __launch_bounds__(SEL_THREADS) k_tree_hist(int64_t n, int L, int64_t C, int shift,
                                                           const int32_t *__restrict__ spl,
                                                           const uint64_t *__restrict__ keys,
                                                           const uint64_t *__restrict__ thr,
                                                           unsigned *__restrict__ ghist)
{
    __shared__ unsigned hist[256];
    const int64_t j = blockIdx.x / C, c = blockIdx.x % C;
    if (spl && !spl[j])
        return;
    int64_t off, m, b, e;
    seg_geom(n, L, j, off, m);
    chunk_range(off, m, C, c, b, e);
    const uint64_t prefix = thr[j];
    const uint64_t mask = shift == 56 ? 0ull : ~0ull << (shift + 8);
    hist[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t p = b + threadIdx.x; p < e; p += SEL_THREADS) {
        const uint64_t k = keys[p];
        if ((k & mask) == prefix)
            atomicAdd(&hist[(k >> shift) & 255], 1u);
    }
    __syncthreads();
    if (hist[threadIdx.x])
        atomicAdd(&ghist[j * 256 + threadIdx.x], hist[threadIdx.x]);
}

__global__ void __launch_bounds__(32) k_tree_digit(int shift, const int32_t *__restrict__ spl,
                                                   uint64_t *__restrict__ thr, int64_t *__restrict__ srank,
                                                   unsigned *__restrict__ ghist)
{
    const int64_t j = blockIdx.x;
    if (spl && !spl[j])
        return;
    unsigned *h = ghist + j * 256;
    int dg;
    int64_t below;
    const int64_t rank = srank[j];
    warp_pick(h, rank, dg, below);
    __syncwarp();
    for (int q = 0; q < 8; q++)
        h[8 * threadIdx.x + q] = 0;
    if (threadIdx.x == 0) {
        thr[j] |= (uint64_t)dg << shift;
        srank[j] = rank - below;
    }
}

// Members with key <= thr[j] (half u) in every chunk of a cluster of several chunks, and their exclusive scan
// over the cluster's chunks (one warp per cluster): where each chunk's u and v members start.
__global__ void __launch_bounds__(SEL_THREADS) k_tree_count(int64_t n, int L, int64_t C,
                                                            const int32_t *__restrict__ spl,
                                                            const uint64_t *__restrict__ keys,
                                                            const uint64_t *__restrict__ thr,
                                                            int32_t *__restrict__ ccount)
{
    __shared__ int wsum[SEL_THREADS / 32];
    const int64_t j = blockIdx.x / C, c = blockIdx.x % C;
    if (spl && !spl[j])
        return;
    int64_t off, m, b, e;
    seg_geom(n, L, j, off, m);
    chunk_range(off, m, C, c, b, e);
    const uint64_t T = thr[j];
    int cnt = 0;
    for (int64_t p = b + threadIdx.x; p < e; p += SEL_THREADS)
        cnt += keys[p] <= T;
    for (int o = 16; o > 0; o >>= 1)
        cnt += __shfl_xor_sync(FULL_MASK, cnt, o);
    if ((threadIdx.x & 31) == 0)
        wsum[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < SEL_THREADS / 32; w++)
            t += wsum[w];
        ccount[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(32) k_tree_cscan(int64_t C, const int32_t *__restrict__ spl,
                                                   const int32_t *__restrict__ ccount, int32_t *__restrict__ cbase)
{
    const int64_t j = blockIdx.x;
    if (spl && !spl[j])
        return;
    const int lane = threadIdx.x;
    int carry = 0;
    for (int64_t c0 = 0; c0 < C; c0 += 32) {
        const int64_t c = c0 + lane;
        const int v = c < C ? ccount[j * C + c] : 0;
        int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL_MASK, incl, o);
            if (lane >= o)
                incl += u;
        }
        if (c < C)
            cbase[j * C + c] = carry + incl - v;
        carry += __shfl_sync(FULL_MASK, incl, 31);
    }
}

// Stable partition of every cluster of depth L, chunk by chunk: the members with key <= thr[j] to the left
// ceil(m/2) positions, the others after them, each in their previous order (cbase: where the chunk's u members
// start among the cluster's, NULL for clusters of one chunk); clusters that do not split are copied.
__global__ void __launch_bounds__(SEL_THREADS) k_tree_split(int64_t n, int L, int64_t C,
                                                            const int32_t *__restrict__ spl,
                                                            const uint64_t *__restrict__ keys,
                                                            const uint64_t *__restrict__ thr,
                                                            const int32_t *__restrict__ cbase,
                                                            const int32_t *__restrict__ perm_in,
                                                            int32_t *__restrict__ perm_out, DevStatus *st)
{
    __shared__ int wsum[SEL_THREADS / 32];
    const int64_t j = blockIdx.x / C, c = blockIdx.x % C;
    int64_t off, m, b, e;
    seg_geom(n, L, j, off, m);
    chunk_range(off, m, C, c, b, e);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (spl && !spl[j]) {
        for (int64_t p = b + tid; p < e; p += SEL_THREADS)
            perm_out[p] = perm_in[p];
        return;
    }
    const uint64_t T = thr[j];
    const int64_t h = (m + 1) / 2;
    int64_t bu = cbase ? cbase[blockIdx.x] : 0;
    int64_t bv = (b - off) - bu;
    for (int64_t t0 = b; t0 < e; t0 += SEL_THREADS) {
        const int64_t p = t0 + tid;
        const bool valid = p < e;
        const uint64_t k = valid ? keys[p] : 0;
        const bool f = valid && k <= T;
        const unsigned bal = __ballot_sync(FULL_MASK, f);
        if (lane == 0)
            wsum[warp] = __popc(bal);
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < SEL_THREADS / 32; w++) {
            before += w < warp ? wsum[w] : 0;
            total += wsum[w];
        }
        const int64_t ru = before + __popc(bal & lanemask_lt());  // u members before this one in the tile
        if (valid) {
            const int64_t dst = f ? off + bu + ru : off + h + bv + (tid - ru);
            if (dst >= off && dst < off + m)
                perm_out[dst] = (int32_t)(uint32_t)k;
            else
                flag_error(st, GK_ERR_INVALID, (unsigned)j);
        }
        const int64_t nvalid = min((int64_t)SEL_THREADS, e - t0);
        bu += total;
        bv += nvalid - total;
        __syncthreads();
    }
}

// Labels: clusters numbered left to right.  Cluster j of the last depth L keeps number j + pre[j], or, when it
// splits (spl[j]), its halves take j + pre[j] and j + pre[j] + 1.  With spl == NULL the depth is complete.
__global__ void __launch_bounds__(SEL_THREADS) k_tree_label(int64_t n, int L, int64_t C,
                                                            const int32_t *__restrict__ spl,
                                                            const int32_t *__restrict__ pre,
                                                            const int32_t *__restrict__ perm,
                                                            int32_t *__restrict__ labels)
{
    const int64_t j = blockIdx.x / C, c = blockIdx.x % C;
    int64_t off, m, b, e;
    seg_geom(n, L, j, off, m);
    chunk_range(off, m, C, c, b, e);
    const bool split = spl && spl[j];
    const int32_t base = (int32_t)j + (spl ? pre[j] : 0);
    const int64_t h = (m + 1) / 2;
    for (int64_t p = b + threadIdx.x; p < e; p += SEL_THREADS) {
        const int id = perm[p];
        if ((unsigned)id < (unsigned)n)
            labels[id] = base + (split && p - off >= h ? 1 : 0);
    }
}

// Depth L such that 2^L <= k < 2^(L + 1): depths 0 .. L - 1 split completely, depth L splits k - 2^L clusters.
int tree_depth(int32_t k)
{
    int L = 0;
    while (((int64_t)2 << L) <= (int64_t)k)
        L++;
    return L;
}

// Pass blocks per cluster at depth L: clusters of up to TR_CHUNK members take one.
int64_t tree_chunks(int64_t n, int L)
{
    const int64_t a1 = (n >> L) + 1;
    return std::max<int64_t>(1, (a1 + TR_CHUNK - 1) / TR_CHUNK);
}

struct TreeBufs {
    int32_t *perm_a, *perm_b, *spl, *pre, *ccount, *cbase;
    uint64_t *keys, *thr;
    int64_t *srank;
    unsigned *ghist;
    Top2 *seeds;
    float *cen;
    unsigned long long *acc;  // limb sums of the clusters of several chunks [2][3][d]; flags, masses [2][d]; counts [2]
    unsigned *flg, *cnts, *colmax, *redo_n, *ticket;
    int64_t *redo_at;
    float *mass;
    uint8_t *halves;
    size_t zero_off, zero_bytes, bytes;
};

TreeBufs tree_carve(void *scratch, int64_t n, int64_t d, int32_t k)
{
    Carver cv{static_cast<char *>(scratch), 0, 0};
    const int Lf = tree_depth(k);
    const int64_t S = (int64_t)1 << Lf;
    int64_t chunks = 1, multi = 1;  // chunk blocks; clusters of several chunks
    for (int L = 0; L <= Lf; L++) {
        const int64_t C = tree_chunks(n, L);
        chunks = std::max(chunks, ((int64_t)1 << L) * C);
        if (C > 1)
            multi = std::max(multi, (int64_t)1 << L);
    }
    TreeBufs B{};
    B.perm_a = cv.take<int32_t>((size_t)n);
    B.perm_b = cv.take<int32_t>((size_t)n);
    B.keys = cv.take<uint64_t>((size_t)n);
    B.cen = cv.take<float>((size_t)S * 2 * (size_t)d);
    B.thr = cv.take<uint64_t>((size_t)S);
    B.srank = cv.take<int64_t>((size_t)S);
    B.spl = cv.take<int32_t>((size_t)S);
    B.pre = cv.take<int32_t>((size_t)S);
    B.seeds = cv.take<Top2>((size_t)chunks);
    B.ccount = cv.take<int32_t>((size_t)chunks);
    B.cbase = cv.take<int32_t>((size_t)chunks);
    B.ghist = cv.take<unsigned>((size_t)multi * 256);
    B.halves = cv.take<uint8_t>((size_t)n);
    B.redo_at = cv.take<int64_t>(REDO_CAP);
    B.zero_off = cv.off;  // from here on zero before the first pass
    B.redo_n = cv.take<unsigned>(1);
    B.ticket = cv.take<unsigned>(1);
    B.colmax = cv.take<unsigned>((size_t)d);
    B.acc = cv.take<unsigned long long>((size_t)multi * 6 * (size_t)d);
    B.flg = cv.take<unsigned>((size_t)multi * 2 * (size_t)d);
    B.mass = cv.take<float>((size_t)multi * 2 * (size_t)d);
    B.cnts = cv.take<unsigned>((size_t)multi * 2);
    B.zero_bytes = cv.off - B.zero_off;
    B.bytes = cv.off;
    return B;
}

// Per depth L (S clusters, C chunk blocks per cluster; spl = NULL when every cluster splits):
//   seeds (2 launches), iters x {pass, centres if C > 1, redo}, keys pass, select (1 launch, or 17 when C > 1),
//   split (1 launch, or 3 when C > 1).
template <typename XT>
cudaError_t tree_run(const XT *X, int64_t n, int d, int64_t ld, int32_t k, int32_t iters, uint64_t seed,
                     int32_t *labels, void *scratch, const TreeBufs &B, DevStatus *st, cudaStream_t s)
{
    cudaError_t e;
    if ((e = set_max_smem((const void *)k_tree_pass<XT, false>, (int)pass_smem<XT>(MAX_D))) != cudaSuccess ||
        (e = set_max_smem((const void *)k_tree_pass<XT, true>, (int)pass_smem<XT>(MAX_D))) != cudaSuccess)
        return e;
    const size_t smem = pass_smem<XT>(d);
    const bool vec = x_vec4(X, d, ld);
    if ((e = cudaMemsetAsync(static_cast<char *>(scratch) + B.zero_off, 0, B.zero_bytes, s)) != cudaSuccess)
        return e;
    if (iters > 0)
        k_tree_colmax<XT><<<dim3((unsigned)std::min<int64_t>((n + 63) / 64, 152 * 8), (unsigned)((d + 127) / 128)), 256, 0,
                            s>>>(X, n, d, ld, vec, B.colmax);
    k_tree_iota<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 8), 256, 0, s>>>(B.perm_a, n);
    const int Lf = tree_depth(k);
    const int64_t r = (int64_t)k - ((int64_t)1 << Lf);
    int32_t *cur = B.perm_a, *nxt = B.perm_b;
    for (int L = 0; L <= Lf; L++) {
        const int32_t *spl = nullptr;
        const int64_t S = (int64_t)1 << L;
        if (L == Lf) {
            if (r == 0)
                break;
            k_tree_plan<<<1, 1024, 0, s>>>(n, L, r, B.spl, B.pre);
            spl = B.spl;
        }
        const int64_t C = tree_chunks(n, L);
        const unsigned SC = (unsigned)(S * C);
        k_tree_seed_part<<<SC, SEL_THREADS, 0, s>>>(n, L, C, cur, spl, seed, B.seeds);
        k_tree_seed_final<XT><<<(unsigned)S, TR_THREADS, 0, s>>>(X, n, d, ld, C, spl, B.seeds, B.cen, st);
        for (int it = 0; it < iters; it++) {
            const RedoList redo{B.redo_n, B.redo_at, (int)std::min<int64_t>(REDO_CAP, C > 1 ? n / C : REDO_CAP)};
            k_tree_pass<XT, false><<<SC, TR_THREADS, smem, s>>>(X, n, d, ld, vec, L, C, cur, spl, B.cen, B.colmax, B.acc,
                                                                B.flg, B.mass, B.cnts, B.halves, B.keys, redo, st);
            const unsigned cb = (unsigned)std::min<int64_t>((S * 2 * d + 255) / 256, 152 * 8);
            if (C > 1)
                k_tree_centres<<<cb, 256, 0, s>>>(S, d, C, spl, B.cen, B.colmax, B.acc, B.flg, B.mass, B.cnts, redo);
            k_tree_redo<XT><<<std::max(152u, cb), 256, 0, s>>>(X, n, d, ld, L, S, C, cur, B.halves, B.cen, B.cnts,
                                                               reinterpret_cast<double *>(B.keys), redo, B.ticket);
        }
        k_tree_pass<XT, true><<<SC, TR_THREADS, smem, s>>>(X, n, d, ld, vec, L, C, cur, spl, B.cen, B.colmax, B.acc, B.flg,
                                                           B.mass, B.cnts, B.halves, B.keys, RedoList{}, st);
        if (C == 1) {
            k_tree_select<<<(unsigned)S, SEL_THREADS, 0, s>>>(n, L, spl, B.keys, B.thr);
            k_tree_split<<<SC, SEL_THREADS, 0, s>>>(n, L, C, spl, B.keys, B.thr, nullptr, cur, nxt, st);
        } else {
            k_tree_sel_init<<<(unsigned)S, SEL_THREADS, 0, s>>>(n, L, spl, B.thr, B.srank, B.ghist);
            for (int shift = 56; shift >= 0; shift -= 8) {
                k_tree_hist<<<SC, SEL_THREADS, 0, s>>>(n, L, C, shift, spl, B.keys, B.thr, B.ghist);
                k_tree_digit<<<(unsigned)S, 32, 0, s>>>(shift, spl, B.thr, B.srank, B.ghist);
            }
            k_tree_count<<<SC, SEL_THREADS, 0, s>>>(n, L, C, spl, B.keys, B.thr, B.ccount);
            k_tree_cscan<<<(unsigned)S, 32, 0, s>>>(C, spl, B.ccount, B.cbase);
            k_tree_split<<<SC, SEL_THREADS, 0, s>>>(n, L, C, spl, B.keys, B.thr, B.cbase, cur, nxt, st);
        }
        std::swap(cur, nxt);
    }
    const int64_t Cf = tree_chunks(n, Lf);
    k_tree_label<<<(unsigned)(((int64_t)1 << Lf) * Cf), SEL_THREADS, 0, s>>>(n, Lf, Cf, r > 0 ? B.spl : nullptr,
                                                                             B.pre, cur, labels);
    return cudaGetLastError();
}

}  // namespace

size_t tree_scratch_bytes(int64_t n, int64_t d, int32_t k) { return tree_carve(nullptr, n, d, k).bytes; }

cudaError_t launch_tree(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, int32_t k, int32_t iters,
                        uint64_t seed, int32_t *labels, void *scratch, DevStatus *st, cudaStream_t s)
{
    const TreeBufs B = tree_carve(scratch, n, d, k);
    if (bf16)
        return tree_run(static_cast<const __nv_bfloat16 *>(X), n, (int)d, ld, k, iters, seed, labels, scratch, B, st, s);
    return tree_run(static_cast<const float *>(X), n, (int)d, ld, k, iters, seed, labels, scratch, B, st, s);
}

}  // namespace gkm
