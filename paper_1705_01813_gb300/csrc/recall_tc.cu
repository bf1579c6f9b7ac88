// Exact nearest neighbours of sampled queries with the pair distances screened
// on the tensor cores (tcgen05, BF16 operands, FP32 accumulation in tensor
// memory) and the survivors recomputed in the canonical FP32 order: the keys
// of the FP32 tile kernel (recall.cu), bit for bit.
//
// k_rc_lossy, k_rc_centre, k_rc_queries prepare the queries: FP32 samples are
// centred on the queries' mean unless every query is a BF16 vector already
// (integers up to 256, say); the centred rows rounded to BF16, their squared
// norms, and for each query the smallest exact distance d0 to the first 32
// entries of its graph row, an upper bound to start from.  The slices share the smallest upper
// bound found so far (bound[], by atomic minimum): on their own each of 38
// slices took its own few minima, and a tile waits for its slowest warp.
//
// k_rc_screen, one CTA per 256 queries and slice of the samples, streams the
// slice in tiles of 128 samples.  Sixteen loader warps copy the rows to shared
// memory three 64-column steps ahead (cp.async, every thread its own vectors),
// centre and round them into stages of the 128-byte swizzle layout, and form
// the rows' norms; one thread issues the two 128 x 128 x 16 MMAs of every
// 16 columns into one of two pairs of TMEM accumulators; eight epilogue warps,
// a thread per query, compare every distance's lower bound with the query's
// smallest upper bound T and append the few samples that pass to the query's
// list.  A query whose list overflows is given up by every slice at once
// (400k x 32 with one column 1,000 times the others, 1,000 queries: 6.6 ms
// when its lists ran on, 3.0 now, 2.2 by the FP32 tiles alone).  The queries'
// operand stays in shared memory where it fits (d <= 128) and is staged beside
// the samples' otherwise.
//
// Bounds.  With x', y' the centred rows, u_y = 2^-8 the BF16 rounding (8
// significant bits: half a unit in the last place; 0 for a row that rounding
// left unchanged), u_x the largest |x' - bf16(x')| / |x'| of the batch's
// queries and G the tensor cores' product,
// D = |x'|^2 + |y'|^2 - 2 G is within
//   E = 1.02 [|x'| |y'| (2 (u_x + u_y + u_x u_y) + 8 (d + 2) 2^-24)
//             + (2 d + 16) 2^-23 (|x'|^2 + |y'|^2)]
// of the canonical FP32 distance: rounding of the operands, accumulation of G
// (16-deep steps aligned to their largest term), and the FP32 rounding of the
// centring, the norms, the canonical sum and this comparison.  A query whose
// norm or d0 is not of ordinary size (NaN, infinity, above 1e30, a norm below
// 1e-25, where the bound's relative terms end), whose list overflows or stays
// empty goes to the FP32 tile kernel instead.
//
// More than RC_BATCH queries are screened in batches that reuse the buffers: a
// list takes 8 KB, and all samples of a million as queries would need 8.4 GB.
//
// What bounds it: instruction issue, in the epilogue (two packed FMAs and a
// minimum for two pairs) and the loaders' conversion about alike.  1,000
// queries against 1M x 128 FP32 take 0.71 ms in all; the FP32 tiles took 16.1 ms, bound
// by shared memory at 24 TFLOP/s.  Loads one step ahead in registers, and the
// pass test unrolled over the accumulators in registers (spilled, and three
// roles' code beyond the instruction cache), took 2.0 ms.
#include "common.cuh"
#include "merge.cuh"
#include "recall.cuh"
#include "tc.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

namespace gkm {
namespace {

constexpr int RC_Q = 256;                  // queries per CTA (two MMA tiles)
constexpr int RC_N = 128;                  // samples per tile
constexpr int RC_KB = 64;                  // columns per stage (one 128-byte swizzle row)
constexpr int RC_BLK = 128 * 128;          // bytes of 128 rows of a stage
constexpr int RC_EPI = 8, RC_LOAD = 16;    // epilogue and loader warps; one more issues the MMAs
constexpr int RC_ROWS = RC_N / (2 * RC_LOAD);  // rows of a tile per loader thread (sixteen lanes a row)
constexpr int RC_THREADS = 32 * (RC_EPI + RC_LOAD + 1);
constexpr int RC_RESIDENT = 2;             // K-blocks up to which the queries stay in shared memory
constexpr int RC_STAGES = 3, RC_STAGES_A = 2;  // operand stages: samples only, samples and queries
constexpr int RC_AHEAD = 3;                // steps of raw rows in flight
constexpr int RC_CAP = 2048;               // list entries per query
constexpr int RC_BATCH = 38 * RC_Q;        // queries screened at once, at most (four slices fill the chip): 80 MB of lists
constexpr uint32_t RC_WAIT_ITERS = 1u << 20;
constexpr uint32_t RC_TMEM = 512;          // two buffers x two query tiles x 128 columns

constexpr float RC_U = 1.f / 256.f;  // BF16 rounding (8 significant bits), relative

struct RcBars {
    uint64_t full[RC_STAGES], empty[RC_STAGES], acc_full[2], acc_empty[2], nrm_full[2], fin;
    uint32_t tmem;
    int abort;
};

__host__ __device__ constexpr int rc_stages(int nkb) { return nkb <= RC_RESIDENT ? RC_STAGES : RC_STAGES_A; }
constexpr int RC_RAW = RC_ROWS * 32 * RC_LOAD * 16;  // bytes of a step's raw rows (FP32; BF16 uses half)

size_t rc_smem(int nkb)
{
    return 1024 + (nkb <= RC_RESIDENT ? (size_t)(2 * nkb + RC_STAGES) * RC_BLK : (size_t)3 * RC_STAGES_A * RC_BLK) +
           RC_AHEAD * (size_t)RC_RAW + sizeof(float) * 4 * RC_N + sizeof(RcBars);
}

// cp.async of 16 (FP32) or 8 (BF16) bytes, zeros where !in
template <typename XT>
__device__ __forceinline__ void rc_copy(void *dst, const XT *src, bool in)
{
    const uint32_t a = tc::smem_addr(dst), bytes = in ? 4 * sizeof(XT) : 0;
    if constexpr (sizeof(XT) == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(a), "l"(src), "r"(bytes) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(a), "l"(src), "r"(bytes) : "memory");
}

// pair_d2_seq by one thread with its loads ahead of the sum (vec: 16 or 8 bytes each).
template <typename XT>
__device__ __forceinline__ float pair_d2(const XT *__restrict__ a, const XT *__restrict__ b, int d, bool vec)
{
    if (!vec)
        return pair_d2_seq(a, b, d);
    float acc = 0.f;
#pragma unroll 4
    for (int t = 0; t < d; t += 4) {
        const float4 x = ldx4<XT>(a + t), y = ldx4<XT>(b + t);
        const float e0 = x.x - y.x, e1 = x.y - y.y, e2 = x.z - y.z, e3 = x.w - y.w;
        acc = fmaf(e0, e0, acc);
        acc = fmaf(e1, e1, acc);
        acc = fmaf(e2, e2, acc);
        acc = fmaf(e3, e3, acc);
    }
    return acc;
}

// Any coordinate of a query that BF16 does not hold exactly?
template <typename XT>
__global__ void __launch_bounds__(256) k_rc_lossy(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                  const int32_t *__restrict__ queries, int m, int *__restrict__ lossy)
{
    const int q = blockIdx.x * 8 + (threadIdx.x >> 5);
    bool any = false;
    if (q < m) {
        const int i = queries[q];
        if (i >= 0 && i < n)
            for (int t = lane_id(); t < d; t += 32) {
                const float x = ldx(X + (int64_t)i * ld + t);
                any |= __bfloat162float(__float2bfloat16_rn(x)) != x;
            }
    }
    if (__any_sync(FULL_MASK, any) && lane_id() == 0)
        *lossy = 1;
}

// The centre: the mean of (at most 256 of) the queries, or zero when no query is lossy.  cols: padded columns.
template <typename XT>
__global__ void __launch_bounds__(128) k_rc_centre(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                   const int32_t *__restrict__ queries, int m,
                                                   const int *__restrict__ lossy, float *__restrict__ centre, int cols)
{
    const int t = blockIdx.x * 128 + threadIdx.x;
    if (t >= cols)
        return;
    float s = 0.f;
    int cnt = 0;
    if (*lossy && t < d) {
        const int step = (m + 255) / 256;
#pragma unroll 8
        for (int q = 0; q < m; q += step) {
            const int i = queries[q];
            if (i >= 0 && i < n) {
                s += ldx(X + (int64_t)i * ld + t);
                cnt++;
            }
        }
    }
    s = cnt > 0 ? s / (float)cnt : 0.f;
    centre[t] = isfinite(s) ? s : 0.f;
}

// A query's shared upper bound, as the bits of its float, above zero; RC_NONE for a query that is not screened (any more).
constexpr unsigned RC_NONE = 0u;
__device__ __forceinline__ unsigned rc_bound(float v) { return __float_as_uint(fmaxf(v, 1.17549435e-38f)); }

// One warp per (padded) query: its centred BF16 row, its squared norm and d0 (negative: take the FP32 tiles); and the
// screened queries' largest rounding error relative to their norms (u_x of the bound), as the bits of its float.  The
// differences are exact; 1.001 covers the sums' rounding, 1e-40 what squares lose below FP32's normal range.  On ordinary
// rows u_x is about 0.4 of the 2^-8 that holds for any row, and fewer samples pass: Gaussian 146k x 64, 500 queries
// 239 -> 226 us, 7,841 x 960 in [0, 1], 1,000 queries 321 -> 284.
template <typename XT>
__global__ void __launch_bounds__(256) k_rc_queries(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                    const int32_t *__restrict__ queries, int m,
                                                    const int32_t *__restrict__ g_idx, int kappa,
                                                    const float *__restrict__ centre, int cols, bool vec,
                                                    __nv_bfloat16 *__restrict__ Aq, float2 *__restrict__ info,
                                                    unsigned *__restrict__ bound, int *__restrict__ rounding)
{
    const int q = blockIdx.x * 8 + (threadIdx.x >> 5), lane = lane_id();
    const int i = q < m ? queries[q] : -1;
    const bool in = i >= 0 && i < n;
    float nrm = 0.f, err = 0.f;
    bool any = false;
    for (int t = lane; t < cols; t += 32) {
        const float x = in && t < d ? ldx(X + (int64_t)i * ld + t) - centre[t] : 0.f;
        const __nv_bfloat16 b = __float2bfloat16_rn(x);
        Aq[(int64_t)q * cols + t] = b;
        const float e = __bfloat162float(b) - x;
        any |= e != 0.f;
        err = fmaf(e, e, err);
        nrm = fmaf(x, x, nrm);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nrm += __shfl_xor_sync(FULL_MASK, nrm, o);
        err += __shfl_xor_sync(FULL_MASK, err, o);
    }
    any = __any_sync(FULL_MASK, any);
    // a lane per neighbour (one takes no longer than all 32): a graph whose first entry is poor has a better one
    float d0 = __int_as_float(0x7f800000);
    if (in && lane < kappa) {
        const int j = g_idx[(int64_t)i * kappa + lane];
        if (j >= 0 && j < n && j != i) {
            const float dj = pair_d2(X + (int64_t)i * ld, X + (int64_t)j * ld, d, vec);
            d0 = dj >= 0.f ? dj : d0;  // not a NaN
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        d0 = fminf(d0, __shfl_xor_sync(FULL_MASK, d0, o));
    if (lane != 0 || q >= m)
        return;
    if (!(in && nrm > 1e-25f && nrm < 1e30f && d0 < 1e30f))
        d0 = -1.f;
    else if (any)
        atomicMax(rounding, __float_as_int(fminf(RC_U, 1.001f * sqrtf((1.001f * err + 1e-40f) / nrm))));
    info[q] = make_float2(nrm, d0);
    bound[q] = d0 < 0.f ? RC_NONE : rc_bound(d0);
}

// The bounded wait of one role: gives up when another role has, or after RC_WAIT_ITERS polls.
__device__ __forceinline__ bool rc_wait(uint64_t *bar, uint32_t parity, volatile int *abort)
{
    for (uint32_t it = 0; it < RC_WAIT_ITERS; it++) {
        if (tc::mbar_try_wait(bar, parity))
            return true;
        if (*abort)
            return false;
    }
    *abort = 1;
    return false;
}

template <typename XT>
__global__ void __launch_bounds__(RC_THREADS, 1) k_rc_screen(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                             bool vec, const int32_t *__restrict__ queries, int m,
                                                             const __nv_bfloat16 *__restrict__ Aq,
                                                             const float2 *__restrict__ info,
                                                             const float *__restrict__ centre,
                                                             const int *__restrict__ rounding, int nkb,
                                                             unsigned *__restrict__ bound,
                                                             int32_t *__restrict__ list, int32_t *__restrict__ cnt,
                                                             DevStatus *st)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                            ~static_cast<uintptr_t>(1023));
    const bool resident = nkb <= RC_RESIDENT;
    const int nst = rc_stages(nkb), stage_bytes = resident ? RC_BLK : 3 * RC_BLK;
    unsigned char *ares = base;                                            // resident queries: [K-block][tile]
    unsigned char *ring = base + (resident ? nkb * 2 * RC_BLK : 0);        // stages: samples (, queries' two tiles)
    unsigned char *raw = ring + nst * stage_bytes;                         // raw rows, RC_AHEAD steps
    float *njn = reinterpret_cast<float *>(raw + RC_AHEAD * RC_RAW);       // [2][RC_N]: |y'|^2 less its bound term
    float *njw = njn + 2 * RC_N;                                           // [2][RC_N]: the bound factor times |y'|
    RcBars *B = reinterpret_cast<RcBars *>(njw + 2 * RC_N);
    volatile int *abort = &B->abort;
    const int tid = threadIdx.x, w = tid >> 5, lane = lane_id();
    const int cols = nkb * RC_KB;
    const int q0 = blockIdx.x * RC_Q;
    const int64_t tiles = (n + RC_N - 1) / RC_N;
    const int64_t t_lo = tiles * blockIdx.y / gridDim.y, t_hi = tiles * (blockIdx.y + 1) / gridDim.y;
    const int ntile = (int)(t_hi - t_lo);

    if (w == RC_EPI + RC_LOAD) {
        tc::tmem_alloc(&B->tmem, RC_TMEM);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < nst; s++) {
            tc::mbar_init(&B->full[s], RC_LOAD);
            tc::mbar_init(&B->empty[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            tc::mbar_init(&B->acc_full[b], 1);
            tc::mbar_init(&B->acc_empty[b], RC_EPI);
            tc::mbar_init(&B->nrm_full[b], RC_LOAD);
        }
        tc::mbar_init(&B->fin, 1);
        tc::fence_mbar_init();
        B->abort = 0;
    }
    // 16 bytes of the queries' operand: row (0 .. 255), K-block, 16-byte chunk of its 64 columns
    auto a_chunk = [&](int row, int kb, int ch) {
        return __ldg(reinterpret_cast<const uint4 *>(Aq + (int64_t)(q0 + row) * cols + kb * RC_KB + ch * 8));
    };
    auto a_offset = [](int row, int ch) { return (row >> 7) * RC_BLK + (row & 127) * 128 + ((ch ^ (row & 7)) << 4); };
    if (resident) {
        for (int e = tid; e < nkb * RC_Q * 8; e += RC_THREADS) {
            const int kb = e / (RC_Q * 8), row = (e >> 3) & (RC_Q - 1), ch = e & 7;
            *reinterpret_cast<uint4 *>(ares + kb * 2 * RC_BLK + a_offset(row, ch)) = a_chunk(row, kb, ch);
        }
        tc::fence_proxy_async_smem();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = B->tmem;
    // the factor of |x'| |y'| in E for a row that rounding leaves unchanged, and for one that it changes
    const float u_q = __int_as_float(*rounding);
    const float acc = 8.f * (float)(d + 2) * 5.9604645e-8f;
    const float f_exact = 1.02f * (2.f * u_q + acc), f_lossy = 1.02f * (2.f * (u_q + RC_U + u_q * RC_U) + acc);
    const float c2 = 1.02f * (float)(2 * d + 16) * 1.1920929e-7f;

    if (w < RC_EPI) {
        // ---- epilogue: query q of the block, TMEM lane q % 128 of tile q / 128 ----
        const int ql = (w >> 2) * 128 + (w & 3) * 32 + lane, q = q0 + ql;
        const int self = q < m ? queries[q] : -1;
        const float2 inf = q < m ? info[q] : make_float2(0.f, -1.f);
        const float s_q = sqrtf(inf.x), n_q = inf.x * (1.f - c2);
        // low + n_q <= smallest upper bound; a query that is not screened passes nothing
        const float none = -__int_as_float(0x7f800000);
        float T = inf.y >= 0.f ? inf.y - n_q : none;
        const uint32_t lane_addr = taddr + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)((w >> 2) * 128);
        for (int ti = 0; ti < ntile; ti++) {
            const int buf = ti & 1;
            const uint32_t ph = (uint32_t)(ti >> 1) & 1u;
            const unsigned shared = q < m ? __ldcg(bound + q) : RC_NONE;  // arrives during the wait
            const bool ok = rc_wait(&B->nrm_full[buf], ph, abort) && rc_wait(&B->acc_full[buf], ph, abort);
            if (!__all_sync(FULL_MASK, ok))
                break;
            tc::fence_after_sync();
            T = shared == RC_NONE ? none : fminf(T, __uint_as_float(shared) - n_q);
            const float before = T;
            const float *nb = njn + buf * RC_N, *wb = njw + buf * RC_N;
            const float2 m2 = make_float2(-2.f, -2.f), ms = make_float2(-s_q, -s_q);
            for (int c0 = 0; c0 < RC_N; c0 += 32) {
                float g[32];
                const uint32_t col = lane_addr + (uint32_t)(buf * 256 + c0);
                __syncwarp();
                tc::tmem_ld32(col, g);
                tc::tmem_ld_wait();
                float low = __int_as_float(0x7f800000);
#pragma unroll
                for (int c = 0; c < 32; c += 4) {
                    const float4 p = *reinterpret_cast<const float4 *>(nb + c0 + c);
                    const float4 v = *reinterpret_cast<const float4 *>(wb + c0 + c);
                    const float2 l0 = __ffma2_rn(ms, make_float2(v.x, v.y),
                                                 __ffma2_rn(m2, make_float2(g[c], g[c + 1]), make_float2(p.x, p.y)));
                    const float2 l1 = __ffma2_rn(ms, make_float2(v.z, v.w),
                                                 __ffma2_rn(m2, make_float2(g[c + 2], g[c + 3]), make_float2(p.z, p.w)));
                    low = fminf(low, fminf(fminf(l0.x, l0.y), fminf(l1.x, l1.y)));
                }
                if (!__any_sync(FULL_MASK, low <= T))
                    continue;
                // some query of the warp takes one of these samples: again, column by column
                const int64_t j0 = (t_lo + ti) * RC_N + c0;
                // (the upper bounds come first, so that a slice that starts from a loose T appends only what is near
                // its minimum; an upper bound is 2 E above the lower one, E's norm term being c2 (n_q + n_j))
                auto lower = [&](int c) {
                    __syncwarp();
                    return fmaf(-s_q, wb[c0 + c], fmaf(-2.f, tc::tmem_ld1(col + (uint32_t)c), nb[c0 + c]));
                };
                auto append = [&](int c) {
                    const int at = atomicAdd(cnt + q, 1);
                    if (at < RC_CAP)
                        list[(int64_t)q * RC_CAP + at] = (int32_t)(j0 + c);
                    else  // a query of the FP32 tiles: no slice needs to look at it again
                        T = none;
                };
                unsigned hits = 0;
#pragma unroll 1
                for (int c = 0; c < 32; c++) {
                    const float l = lower(c);
                    if (l <= T && (int)(j0 + c) != self && q < m) {
                        hits |= 1u << c;
                        T = fminf(T, l + 2.f * s_q * wb[c0 + c] + 2.1f * c2 * (inf.x + nb[c0 + c]));
                    }
                }
                if (__any_sync(FULL_MASK, __popc(hits) > 1)) {  // some passed only the bound before the last one
#pragma unroll 1
                    for (int c = 0; c < 32; c++) {
                        const float l = lower(c);
                        if (((hits >> c) & 1u) && l <= T)
                            append(c);
                    }
                } else if (hits) {
                    append(__ffs(hits) - 1);
                }
            }
            if (T < before)  // rounded up: the sum's own rounding
                atomicMin(bound + q, T == none ? RC_NONE : rc_bound((T + n_q) * 1.000001f));
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0)
                tc::mbar_arrive(&B->acc_empty[buf]);
        }
    } else if (w < RC_EPI + RC_LOAD) {
        // ---- loaders: sixteen lanes per row, each four consecutive columns of a step ----
        const int lt = tid - 32 * RC_EPI, lw = lt >> 5, sub = lane & 15, rsel = lane >> 4;
        constexpr int VB = 4 * (int)sizeof(XT);  // bytes of a thread's raw vector
        // step g: K-block g % nkb of tile g / nkb, into slot g % RC_AHEAD
        int f_tile = 0, f_kb = 0, f_slot = 0;
        auto fetch = [&]() {
            if (f_tile < ntile) {
                const int col = f_kb * RC_KB + sub * 4;
                unsigned char *dst = raw + f_slot * RC_RAW + lt * VB;
#pragma unroll
                for (int it = 0; it < RC_ROWS; it++) {
                    const int64_t j = (t_lo + f_tile) * RC_N + it * 2 * RC_LOAD + lw * 2 + rsel;
                    const bool in = j < n && col < d;
                    const XT *p = X + (in ? j * ld + col : 0);
                    unsigned char *q = dst + it * 32 * RC_LOAD * VB;
                    if (vec) {
                        rc_copy<XT>(q, p, in);
                    } else {
                        XT *e = reinterpret_cast<XT *>(q);
#pragma unroll
                        for (int z = 0; z < 4; z++)
                            e[z] = in && col + z < d ? p[z] : XT(0.f);
                    }
                }
                if (++f_kb == nkb) {
                    f_kb = 0;
                    f_tile++;
                }
                f_slot = f_slot + 1 == RC_AHEAD ? 0 : f_slot + 1;
            }
            cp_async_commit();  // a group per step, empty past the last one
        };
        for (int g = 0; g < RC_AHEAD - 1; g++)
            fetch();
        int stage = 0, slot = 0;
        uint32_t ph = 1;  // a fresh barrier's previous phase counts as complete
        bool ok = true;
        for (int ti = 0; ti < ntile && ok; ti++) {
            float ns[RC_ROWS];
            unsigned lossy = 0;
#pragma unroll
            for (int it = 0; it < RC_ROWS; it++)
                ns[it] = 0.f;
            for (int kb = 0; kb < nkb; kb++) {
                fetch();  // the slot read in the previous step
                const int col = kb * RC_KB + sub * 4;
                const float4 c4 = __ldg(reinterpret_cast<const float4 *>(centre + col));
                uint4 aq[RC_Q * 8 / (32 * RC_LOAD)];  // in flight during the wait and the conversion
                if (!resident) {
#pragma unroll
                    for (int e = 0; e < RC_Q * 8 / (32 * RC_LOAD); e++) {
                        const int c = lt + e * 32 * RC_LOAD;
                        aq[e] = a_chunk(c >> 3, kb, c & 7);
                    }
                }
                ok = rc_wait(&B->empty[stage], ph, abort);
                if (!__all_sync(FULL_MASK, ok)) {
                    ok = false;
                    break;
                }
                cp_async_wait<RC_AHEAD - 1>();  // this thread's vectors of this step have arrived
                unsigned char *sb = ring + stage * stage_bytes;
                const unsigned char *src = raw + slot * RC_RAW + lt * VB;
                slot = slot + 1 == RC_AHEAD ? 0 : slot + 1;
#pragma unroll
                for (int it = 0; it < RC_ROWS; it++) {
                    const int r = it * 2 * RC_LOAD + lw * 2 + rsel;
                    float4 v;
                    if constexpr (sizeof(XT) == 4)
                        v = *reinterpret_cast<const float4 *>(src + it * 32 * RC_LOAD * VB);
                    else
                        v = bf16x4_to_float4(*reinterpret_cast<const uint2 *>(src + it * 32 * RC_LOAD * VB));
                    // columns past d are zero in the samples and the centre
                    const float x0 = v.x - c4.x, x1 = v.y - c4.y, x2 = v.z - c4.z, x3 = v.w - c4.w;
                    ns[it] = fmaf(x0, x0, fmaf(x1, x1, fmaf(x2, x2, fmaf(x3, x3, ns[it]))));
                    const __nv_bfloat162 b0 = __floats2bfloat162_rn(x0, x1), b1 = __floats2bfloat162_rn(x2, x3);
                    if constexpr (sizeof(XT) == 4) {  // BF16 holds x exactly when the low half of its word is zero
                        const unsigned low = (__float_as_uint(x0) | __float_as_uint(x1) | __float_as_uint(x2) |
                                              __float_as_uint(x3)) & 0xffffu;
                        lossy |= low ? 1u << it : 0u;
                    }
                    uint2 pk;
                    pk.x = *reinterpret_cast<const uint32_t *>(&b0);
                    pk.y = *reinterpret_cast<const uint32_t *>(&b1);
                    *reinterpret_cast<uint2 *>(sb + r * 128 + (((sub >> 1) ^ (r & 7)) << 4) + (sub & 1) * 8) = pk;
                }
                if (!resident) {
#pragma unroll
                    for (int e = 0; e < RC_Q * 8 / (32 * RC_LOAD); e++) {
                        const int c = lt + e * 32 * RC_LOAD, row = c >> 3, ch = c & 7;
                        *reinterpret_cast<uint4 *>(sb + RC_BLK + a_offset(row, ch)) = aq[e];
                    }
                }
                tc::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0)
                    tc::mbar_arrive(&B->full[stage]);
                if (++stage == nst) {
                    stage = 0;
                    ph ^= 1u;
                }
            }
            if (!ok)
                break;
            // the rows' norms and bound factors, for the epilogue
            const int64_t j0 = (t_lo + ti) * RC_N;
            const int buf = ti & 1;
            // sums over the sixteen lanes of a row: two steps that halve the rows a lane holds, two plain ones; lane
            // sub then has row sub / 4 of its four
            static_assert(RC_ROWS == 4, "the exchange below");
            const bool hi = (sub & 8) != 0, hi2 = (sub & 4) != 0;
            float n0 = (hi ? ns[2] : ns[0]) + __shfl_xor_sync(FULL_MASK, hi ? ns[0] : ns[2], 8);
            const float n1 = (hi ? ns[3] : ns[1]) + __shfl_xor_sync(FULL_MASK, hi ? ns[1] : ns[3], 8);
            n0 = (hi2 ? n1 : n0) + __shfl_xor_sync(FULL_MASK, hi2 ? n0 : n1, 4);
            n0 += __shfl_xor_sync(FULL_MASK, n0, 2);
            n0 += __shfl_xor_sync(FULL_MASK, n0, 1);
            unsigned any = 0;  // bit it: rounding changed row it of this lane's half
#pragma unroll
            for (int it = 0; it < RC_ROWS; it++)
                any |= ((__ballot_sync(FULL_MASK, (lossy >> it) & 1u) >> (lane & 16)) & 0xffffu) ? 1u << it : 0u;
            ok = rc_wait(&B->acc_empty[buf], ((uint32_t)(ti >> 1) & 1u) ^ 1u, abort);
            if (!__all_sync(FULL_MASK, ok)) {
                ok = false;
                break;
            }
            if ((sub & 3) == 0) {
                const int it = sub >> 2, r = it * 2 * RC_LOAD + lw * 2 + rsel;
                const bool in = j0 + r < n;
                njn[buf * RC_N + r] = in ? n0 * (1.f - c2) : __int_as_float(0x7f800000);
                njw[buf * RC_N + r] = in ? sqrtf(n0) * ((any >> it) & 1u ? f_lossy : f_exact) : 0.f;
            }
            __syncwarp();
            if (lane == 0)
                tc::mbar_arrive(&B->nrm_full[buf]);
        }
        cp_async_wait_all();
    } else if (lane == 0) {
        // ---- the MMAs ----
        const uint32_t idesc = tc::idesc_bf16_f32(128, RC_N);
        int stage = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int ti = 0; ti < ntile && ok; ti++) {
            const int buf = ti & 1;
            ok = rc_wait(&B->acc_empty[buf], ((uint32_t)(ti >> 1) & 1u) ^ 1u, abort);
            for (int kb = 0; kb < nkb && ok; kb++) {
                ok = rc_wait(&B->full[stage], ph, abort);
                if (!ok)
                    break;
                tc::fence_after_sync();
                const uint32_t sb = tc::smem_addr(ring + stage * stage_bytes);
                const uint32_t sa = resident ? tc::smem_addr(ares + kb * 2 * RC_BLK) : sb + RC_BLK;
#pragma unroll
                for (int mt = 0; mt < 2; mt++)
#pragma unroll
                    for (int s = 0; s < RC_KB / 16; s++)
                        tc::mma_bf16(taddr + (uint32_t)(buf * 256 + mt * 128),
                                     tc::desc_k128(sa + mt * RC_BLK + 32 * s), tc::desc_k128(sb + 32 * s), idesc,
                                     kb > 0 || s > 0);
                tc::mma_commit(&B->empty[stage]);
                if (kb + 1 == nkb)
                    tc::mma_commit(&B->acc_full[buf]);
                if (++stage == nst) {
                    stage = 0;
                    ph ^= 1u;
                }
            }
        }
        if (!ok) {  // a wait gave up: report, and wait (bounded) for the MMAs issued so far
            flag_error(st, GK_ERR_TIMEOUT, (unsigned)blockIdx.x);
            tc::mma_commit(&B->fin);
            tc::mbar_wait_bounded(&B->fin, 0, RC_WAIT_ITERS);
        }
    }
    __syncwarp();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0 && *abort)
        flag_error(st, GK_ERR_TIMEOUT, (unsigned)blockIdx.x);
    if (w == RC_EPI + RC_LOAD)
        tc::tmem_dealloc(taddr, RC_TMEM);
}

// One block per query of a batch that begins at query q0 of the call: the canonical distances of its list, the smallest
// key; a query without a usable list goes to `left` (by its place in the call, counted in *nleft), for the FP32 tiles.
template <typename XT>
__global__ void __launch_bounds__(128) k_rc_exact(const XT *__restrict__ X, int64_t n, int d, int64_t ld, bool vec,
                                                  const int32_t *__restrict__ queries, int m,
                                                  const float2 *__restrict__ info, const int32_t *__restrict__ list,
                                                  const int32_t *__restrict__ cnt, uint64_t *__restrict__ best,
                                                  int q0, int32_t *__restrict__ left, int32_t *__restrict__ nleft)
{
    __shared__ uint64_t s_best[4];
    const int q = blockIdx.x;
    const int c = cnt[q], i = queries[q];
    if (info[q].y < 0.f || c <= 0 || c > RC_CAP) {
        if (threadIdx.x == 0)
            left[atomicAdd(nleft, 1)] = q0 + q;
        return;
    }
    uint64_t k = ~0ull;
    for (int e = threadIdx.x; e < c; e += 128) {
        const int j = list[(int64_t)q * RC_CAP + e];
        k = min(k, pack_key(pair_d2(X + (int64_t)i * ld, X + (int64_t)j * ld, d, vec), j));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        k = min(k, (uint64_t)__shfl_xor_sync(FULL_MASK, (unsigned long long)k, o));
    if (lane_id() == 0)
        s_best[threadIdx.x >> 5] = k;
    __syncthreads();
    if (threadIdx.x == 0)
        best[q] = min(min(s_best[0], s_best[1]), min(s_best[2], s_best[3]));
}

struct RcBufs {
    int *nleft;  // of the call; then, of the batch: lossy, the queries' rounding and the list counters
    int *flags;
    int32_t *cnt, *left, *list;
    float *centre;
    float2 *info;
    unsigned *bound;
    __nv_bfloat16 *Aq;
    size_t bytes;
};

// Queries per batch: the call's, shared out evenly over as few batches as hold them.
int32_t rc_batch(int32_t m)
{
    const int32_t nb = (int32_t)(((int64_t)m + RC_BATCH - 1) / RC_BATCH);
    return (int32_t)((((int64_t)m + nb - 1) / nb + RC_Q - 1) / RC_Q * RC_Q);
}

// Everything but `left` is of one batch, whatever m.
RcBufs rc_carve(void *scratch, int64_t d, int32_t m)
{
    Carver cv{static_cast<char *>(scratch), 0, 0};
    const int64_t cols = (d + RC_KB - 1) / RC_KB * RC_KB;
    const size_t mb = (size_t)std::min(m, RC_BATCH), mp = (mb + RC_Q - 1) / RC_Q * RC_Q;
    RcBufs B{};
    B.nleft = cv.take<int>(64);
    B.flags = cv.take<int>(64);
    B.cnt = cv.take<int32_t>(mb);
    B.left = cv.take<int32_t>((size_t)m);
    B.list = cv.take<int32_t>(mb * RC_CAP);
    B.centre = cv.take<float>((size_t)cols);
    B.info = cv.take<float2>(mb);
    B.bound = cv.take<unsigned>(mb);
    B.Aq = cv.take<__nv_bfloat16>(mp * (size_t)cols);
    B.bytes = cv.off;
    return B;
}

template <typename XT>
cudaError_t screen_t(const XT *X, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx, int32_t kappa,
                     const int32_t *queries, int32_t m, uint64_t *best, void *scratch, const int32_t **left,
                     const int32_t **nleft, DevStatus *st, cudaStream_t s)
{
    const RcBufs B = rc_carve(scratch, d, m);
    const int nkb = (int)((d + RC_KB - 1) / RC_KB), cols = nkb * RC_KB;
    const int64_t tiles = (n + RC_N - 1) / RC_N;
    const int32_t batch = rc_batch(m);
    const bool vec = x_vec4(X, d, ld);
    cudaError_t e;
    if ((e = set_max_smem(reinterpret_cast<const void *>(k_rc_screen<XT>), 227 * 1024)) != cudaSuccess)
        return e;
    for (int64_t q0 = 0; q0 < m; q0 += batch) {
        const int32_t *qs = queries + q0;
        const int mb = (int)std::min<int64_t>(batch, m - q0), qb = (mb + RC_Q - 1) / RC_Q;
        const int64_t slices = std::min<int64_t>(std::max(1, 152 / qb), tiles);
        char *zero = reinterpret_cast<char *>(q0 == 0 ? B.nleft : B.flags);
        if ((e = cudaMemsetAsync(zero, 0, reinterpret_cast<char *>(B.cnt + mb) - zero, s)) != cudaSuccess)
            return e;
        if (std::is_same_v<XT, float>)  // BF16 samples are not rounded
            k_rc_lossy<XT><<<(mb + 7) / 8, 256, 0, s>>>(X, n, (int)d, ld, qs, mb, B.flags);
        k_rc_centre<XT><<<(cols + 127) / 128, 128, 0, s>>>(X, n, (int)d, ld, qs, mb, B.flags, B.centre, cols);
        k_rc_queries<XT><<<qb * RC_Q / 8, 256, 0, s>>>(X, n, (int)d, ld, qs, mb, g_idx, kappa, B.centre, cols, vec, B.Aq,
                                                       B.info, B.bound, B.flags + 1);
        k_rc_screen<XT><<<dim3((unsigned)qb, (unsigned)slices), RC_THREADS, rc_smem(nkb), s>>>(
            X, n, (int)d, ld, vec, qs, mb, B.Aq, B.info, B.centre, B.flags + 1, nkb, B.bound, B.list, B.cnt, st);
        k_rc_exact<XT><<<(unsigned)mb, 128, 0, s>>>(X, n, (int)d, ld, vec, qs, mb, B.info, B.list, B.cnt, best + q0,
                                                    (int)q0, B.left, B.nleft);
    }
    *left = B.left;
    *nleft = B.nleft;
    return cudaGetLastError();
}

}  // namespace

size_t recall_screen_bytes(int64_t d, int32_t m) { return rc_carve(nullptr, d, m).bytes; }

cudaError_t launch_recall_screen(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx,
                                 int32_t kappa, const int32_t *queries, int32_t m, uint64_t *best, void *scratch,
                                 const int32_t **left, const int32_t **nleft, DevStatus *st, cudaStream_t s)
{
    if (bf16)
        return screen_t(static_cast<const __nv_bfloat16 *>(X), n, d, ld, g_idx, kappa, queries, m, best, scratch, left,
                        nleft, st, s);
    return screen_t(static_cast<const float *>(X), n, d, ld, g_idx, kappa, queries, m, best, scratch, left, nleft, st, s);
}

}  // namespace gkm
