// Graph-guided assignment (Alg. 2 candidate loop with the closest-centroid
// rule of Sec. 4.2, "GK-means^-"):
//   Q_i = { L[i] } u { L[G[i][j]] : j < kappa }          (candidate clusters)
//   L'[i] = argmin over r in Q_i of (||x_i - C_r||^2, r)  (ties -> smaller label)
//
// One warp per sample.  The warp collects the distinct labels of the kappa + 1
// candidates (collect_labels) and takes the distances to their centroids; a
// shuffle reduction picks the (distance, label)
// minimum.  Per-block FP64 partial sums of the winning distances and the
// count of changed labels are reduced in a fixed order afterwards, so every
// run gives the same bits.
#include "assign_common.cuh"
#include "common.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

namespace gkm {

bool assign_tc_supported(int64_t d, int64_t ld, const float *X, const float *C, int32_t kappa);
cudaError_t launch_assign_tc(const float *X, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx, int32_t kappa,
                             const float *C, const __nv_bfloat16 *Cb, const float *delta, const float *cnorm,
                             int32_t k, const int32_t *labels_in, const int32_t *members, int32_t *sel_lab,
                             int32_t *sel_n, int32_t *tile_flag, DevStatus *st, cudaStream_t s);

constexpr int AS_WARPS = 8;
constexpr int AS_BLOCKS = 152 * 8;  // fixed grid: the FP64 partial sums have a fixed order
// The row kernels for d <= 128 fit six blocks per SM (at most 40 registers a thread: more warps in flight
// for the latency-bound centroid gathers), those for d <= 256 five (the FP32 one spills at 40: 400k x 256 1003 us at
// six, 895 at five).  Every row kernel runs on a grid of the blocks resident at once
// (resident_grid), one wave; the distortion sums do not depend on it: k_assign_reduce forms them on its
// own fixed grid.
constexpr int AS_ROWS_PER_SM = 6;
constexpr int AS_QCAP = MAX_KAPPA + 1;
constexpr int AS_TILE = 128;  // samples per tile of the tensor-core assignment

constexpr int AS_G = 8;
constexpr int AS_HASH = 256;                                  // slots of the per-warp label set
constexpr int AS_QROW = (AS_QCAP + AS_G + 3) / 4 * 4;         // candidate list row, padding included
static_assert(AS_HASH > AS_QCAP, "the label set must never fill up");

// The distinct candidate labels of sample i in list order (the own label first, then the neighbours'), written to
// qlist; returns their number.  Repeats are dropped with __match_any_sync inside each batch of 32 and, across batches,
// with a per-warp open-addressing set in shared memory (one atomicCAS per new label).
// SHORT: lists of one batch are expected and spared the set (a test of it costs the wider rows 2%).
template <bool SHORT = false>
__device__ __forceinline__ int collect_labels(int64_t i, int own, const int32_t *__restrict__ G, int kappa, int64_t n,
                                              int k, const int32_t *__restrict__ Lin, int *qlist, int *tab,
                                              DevStatus *st)
{
    const int lane = lane_id(), ncand = kappa + 1;
    const bool several = !SHORT || ncand > 32;
    if (several) {
#pragma unroll
        for (int q = lane * 4; q < AS_HASH; q += 128)
            *reinterpret_cast<int4 *>(tab + q) = make_int4(-1, -1, -1, -1);
        __syncwarp();
    }
    int u = 0;
    for (int c0 = 0; c0 < ncand; c0 += 32) {
        int c = c0 + lane;
        int lab = -1;
        if (c == 0) {
            lab = own;
        } else if (c < ncand) {
            int nb = __ldcs(G + i * kappa + (c - 1));
            if ((unsigned)nb < (unsigned)n)
                lab = Lin[nb];
            else
                flag_error(st, GK_ERR_INVALID, (unsigned)i);
        }
        if (c < ncand && (unsigned)lab >= (unsigned)k) {
            flag_error(st, GK_ERR_INVALID, (unsigned)i);
            lab = -1;
        }
        const unsigned peers = __match_any_sync(FULL_MASK, lab);
        bool fresh = lab >= 0 && (peers & lanemask_lt()) == 0u;
        if (fresh && several) {
            fresh = false;
            unsigned h = ((unsigned)lab * 0x9E3779B1u) >> 24;  // 8-bit multiplicative hash
            for (int probe = 0; probe < AS_HASH; probe++) {    // the set is never full: ends early
                const int old = atomicCAS(tab + h, -1, lab);
                if (old == -1) {
                    fresh = true;
                    break;
                }
                if (old == lab)
                    break;
                h = (h + 1) & (AS_HASH - 1);
            }
        }
        const unsigned fr = __ballot_sync(FULL_MASK, fresh);
        if (fresh)
            qlist[u + __popc(fr & lanemask_lt())] = lab;
        u += __popc(fr);
    }
    __syncwarp();
    return u;
}

// The same without a set: repeats across batches are looked for in the list.  For k_assign, whose lanes walk centroid
// rows of their own and live on L1, of which the sets would take 8 KB a block (300k x 130 2500 us an assignment with
// them, 2240 without).
__device__ __forceinline__ int collect_labels_plain(int64_t i, int own, const int32_t *__restrict__ G, int kappa,
                                                    int64_t n, int k, const int32_t *__restrict__ Lin, int *qlist,
                                                    DevStatus *st)
{
    const int lane = lane_id(), ncand = kappa + 1;
    int u = 0;
    for (int c0 = 0; c0 < ncand; c0 += 32) {
        const int c = c0 + lane;
        int lab = -1;
        if (c == 0) {
            lab = own;
        } else if (c < ncand) {
            const int nb = __ldcs(G + i * kappa + (c - 1));
            if ((unsigned)nb < (unsigned)n)
                lab = Lin[nb];
            else
                flag_error(st, GK_ERR_INVALID, (unsigned)i);
        }
        if (c < ncand && (unsigned)lab >= (unsigned)k) {
            flag_error(st, GK_ERR_INVALID, (unsigned)i);
            lab = -1;
        }
        const unsigned peers = __match_any_sync(FULL_MASK, lab);
        bool fresh = lab >= 0 && (peers & lanemask_lt()) == 0u;
        for (int q = 0; q < u && fresh; q++)
            fresh = qlist[q] != lab;
        const unsigned fr = __ballot_sync(FULL_MASK, fresh);
        if (fresh)
            qlist[u + __popc(fr & lanemask_lt())] = lab;
        u += __popc(fr);
        __syncwarp();
    }
    return u;
}

// Several assignments of the same samples in a row (Track): a sample whose graph row and own centroid are as they were
// in the previous one still has its distance best[i] to that centroid, which every other candidate with an unchanged
// centroid lost to then (its cluster has the same members, so it was a candidate then too); only candidates of changed
// clusters can win now.  The result, and every bit of best[], is that of the whole evaluation.
//
// k_assign_select sorts the samples by what they need: none of a known sample's neighbours is in a changed cluster:
// its label is written and it is done; otherwise it goes to the back list (candidates of changed clusters only), and a
// sample whose own centroid or graph row changed goes to the front list (all candidates).  The assignment kernels then
// walk the lists.  Doing the test inside them cost registers that the evaluation needs: 30 -> 32 ms for the 1M x 128
// graph construction, where almost no sample is done early (this kernel: 13 us of 1 ms there).  The lists' order
// varies from call to call and decides nothing but which warp takes a sample.  A neighbour costs one byte gather, of
// the mark that k_assign_reduce left for its cluster (its label and then the cluster's byte, 0.52 ms at 2M x 40: the
// L1's one lookup a cycle). Against evaluating everything: a fit of 2M x 512 BF16 (k = 200,000) takes 1.0 ms an
// assignment instead of 9.0 once its labels have settled.
constexpr int SL_WARPS = 8;

template <int S>
__global__ void __launch_bounds__(SL_WARPS * 32) k_assign_select(int64_t n, const int32_t *__restrict__ G, int kappa,
                                                                 int k, const int32_t *__restrict__ Lin,
                                                                 int32_t *__restrict__ Lout, const Track trk,
                                                                 int32_t *__restrict__ todo)
{
    constexpr int B = S <= 2 ? 4 : 2;  // samples whose neighbours are looked up together, S slots of 32 each
    __shared__ int s_n[2], s_at[2];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int64_t step = (int64_t)gridDim.x * SL_WARPS * 32;
    for (int64_t b0 = (int64_t)blockIdx.x * SL_WARPS * 32; b0 < n; b0 += step) {
        const int64_t i0 = b0 + w * 32, i = i0 + lane;
        int own = -1;
        bool known = false;
        if (i < n) {
            own = Lin[i];
            known = trk.mark[i] == 0;  // a label out of range is marked
            if (trk.row_changed && trk.row_changed[i]) {
                trk.row_changed[i] = 0;
                known = false;
            }
        }
        unsigned left = __ballot_sync(FULL_MASK, known);
        unsigned touched = 0;  // known samples with a neighbour in a changed cluster (or an id out of range)
        while (left) {
            int src[B];
            int nb[B][S];
#pragma unroll
            for (int q = 0; q < B; q++) {
                src[q] = left ? __ffs(left) - 1 : -1;
                left &= left - 1;
#pragma unroll
                for (int u = 0; u < S; u++) {
                    const int c = lane + 32 * u;
                    nb[q][u] = src[q] >= 0 && c < kappa ? __ldcs(G + (i0 + src[q]) * kappa + c) : -2;
                }
            }
#pragma unroll
            for (int q = 0; q < B; q++)
#pragma unroll
                for (int u = 0; u < S; u++)
                    if (nb[q][u] != -2)
                        nb[q][u] = (unsigned)nb[q][u] < (unsigned)n ? trk.mark[nb[q][u]] : 1;
#pragma unroll
            for (int q = 0; q < B; q++) {
                bool any = false;
#pragma unroll
                for (int u = 0; u < S; u++)
                    any |= nb[q][u] > 0;
                if (__any_sync(FULL_MASK, any) && src[q] >= 0)
                    touched |= 1u << src[q];
            }
        }
        const bool part = known && ((touched >> lane) & 1u) != 0, full = i < n && !known;
        if (known && !part)
            Lout[i] = own;
        // places in the two lists, one atomic per block and list
        if (threadIdx.x < 2)
            s_n[threadIdx.x] = 0;
        __syncthreads();
        const unsigned bf = __ballot_sync(FULL_MASK, full), bp = __ballot_sync(FULL_MASK, part);
        int wf = 0, wp = 0;
        if (lane == 0) {
            wf = atomicAdd(&s_n[0], __popc(bf));
            wp = atomicAdd(&s_n[1], __popc(bp));
        }
        __syncthreads();
        if (threadIdx.x < 2)
            s_at[threadIdx.x] = s_n[threadIdx.x] ? atomicAdd(trk.todo_n + threadIdx.x, s_n[threadIdx.x]) : 0;
        __syncthreads();
        wf = __shfl_sync(FULL_MASK, wf, 0) + s_at[0];
        wp = __shfl_sync(FULL_MASK, wp, 0) + s_at[1];
        if (full)
            todo[wf + __popc(bf & lanemask_lt())] = (int32_t)i;
        else if (part)
            todo[n - 1 - (wp + __popc(bp & lanemask_lt()))] = (int32_t)i;
        __syncthreads();
    }
}

// The samples of an assignment kernel: all of them, or the two lists; f(sample, std::true_type) for the back list.
// (Taking all samples in their order where the lists hold 7/8 of them gained 1% at 1M x 128 and lost 5% at
// 200k x 960 and 2M x 512, where the back list is long.)
template <bool LISTS, typename F>
__device__ __forceinline__ void each_sample(int64_t first, int64_t step, int64_t n, const Track &trk,
                                            const int32_t *__restrict__ todo, F f)
{
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *trk.ticket = 0u;  // for k_assign_reduce
    if constexpr (!LISTS) {
        for (int64_t i = first; i < n; i += step)
            f(i, std::false_type{});
    } else {
        const int nf = trk.todo_n[0], np = trk.todo_n[1];
        int32_t nxt = first < nf ? todo[first] : 0;  // the entries are loaded a sample ahead
        for (int64_t p = first; p < nf; p += step) {
            const int64_t i = nxt;
            if (p + step < nf)
                nxt = todo[p + step];
            f(i, std::false_type{});
        }
        for (int64_t p = first; p < np; p += step)
            f((int64_t)todo[n - 1 - p], std::true_type{});
    }
}

// The candidates of changed clusters among the u of a sample whose own distance is known, moved to the list's front.
__device__ __forceinline__ int track_filter(const Track &trk, int *qlist, int u)
{
    const int lane = lane_id();
    int m = 0;
    for (int c0 = 0; c0 < u; c0 += 32) {
        const int c = c0 + lane;
        const int lab = c < u ? qlist[c] : -1;
        const bool keep = c > 0 && c < u && trk.dirty[lab] != 0;  // entry 0 is the own label
        const unsigned bal = __ballot_sync(FULL_MASK, keep);      // every lane has read its entry
        if (keep)
            qlist[m + __popc(bal & lanemask_lt())] = lab;
        m += __popc(bal);
    }
    __syncwarp();
    return m;
}

// The winner (bd, br) of sample i, written by lane 0.  Without a valid candidate (br still INT_MAX) the input label
// stays, with distance 0, and its cluster counts as changed, so that the next assignment looks again.
__device__ __forceinline__ void write_winner(int64_t i, const int32_t *__restrict__ Lin, int k, float bd, int br,
                                             int32_t *__restrict__ Lout, float *__restrict__ best, const Track &trk)
{
    if (lane_id() != 0)
        return;
    const int own = Lin[i];
    bool changed = br != own;
    if (br == 0x7fffffff) {
        br = own, bd = 0.f;
        changed = true;
    }
    Lout[i] = br;
    if (best)
        best[i] = bd;
    if (changed && trk.dirty_out) {
        if ((unsigned)own < (unsigned)k)
            trk.dirty_out[own] = 1;
        if ((unsigned)br < (unsigned)k)
            trk.dirty_out[br] = 1;
    }
}

template <int VEC>
__device__ __forceinline__ float cand_d2(const float *__restrict__ xs, const float *__restrict__ c, int d);

template <>
__device__ __forceinline__ float cand_d2<4>(const float *__restrict__ xs, const float *__restrict__ c, int d)
{
    const float4 *x4 = reinterpret_cast<const float4 *>(xs);
    const float4 *c4 = reinterpret_cast<const float4 *>(c);
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    const int nv = d >> 2;
#pragma unroll 4
    for (int t = 0; t < nv; t++) {
        float4 xv = x4[t];
        float4 cv = __ldg(c4 + t);
        float e0 = xv.x - cv.x, e1 = xv.y - cv.y, e2 = xv.z - cv.z, e3 = xv.w - cv.w;
        a0 = fmaf(e0, e0, a0);
        a1 = fmaf(e1, e1, a1);
        a2 = fmaf(e2, e2, a2);
        a3 = fmaf(e3, e3, a3);
    }
    return (a0 + a1) + (a2 + a3);
}

template <>
__device__ __forceinline__ float cand_d2<1>(const float *__restrict__ xs, const float *__restrict__ c, int d)
{
    float a0 = 0.f, a1 = 0.f;
    int t = 0;
    for (; t + 1 < d; t += 2) {
        float e0 = xs[t] - __ldg(c + t), e1 = xs[t + 1] - __ldg(c + t + 1);
        a0 = fmaf(e0, e0, a0);
        a1 = fmaf(e1, e1, a1);
    }
    if (t < d) {
        float e0 = xs[t] - __ldg(c + t);
        a0 = fmaf(e0, e0, a0);
    }
    return a0 + a1;
}

template <int VEC, typename XT, bool LISTS>
__global__ void __launch_bounds__(AS_WARPS * 32) k_assign(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                          const int32_t *__restrict__ G, int kappa,
                                                          const float *__restrict__ C, int k,
                                                          const int32_t *__restrict__ Lin,
                                                          int32_t *__restrict__ Lout, float *__restrict__ best_out,
                                                          DevStatus *st, const Track trk,
                                                          const int32_t *__restrict__ todo)
{
    extern __shared__ __align__(16) float smem[];
    const int w = threadIdx.x >> 5, lane = lane_id();
    const int dpad = (d + 3) & ~3;
    float *xs = smem + w * dpad;
    int *qlist = reinterpret_cast<int *>(smem + AS_WARPS * dpad) + w * AS_QCAP;

    each_sample<LISTS>((int64_t)blockIdx.x * AS_WARPS + w, (int64_t)gridDim.x * AS_WARPS, n, trk, todo,
                       [&](int64_t i, auto part) {
        constexpr bool PART = decltype(part)::value;
        // stage x_i
        const XT *xi = X + i * ld;
        if (VEC == 4) {
            for (int t = lane; t < (d >> 2); t += 32)
                reinterpret_cast<float4 *>(xs)[t] = ldx4<XT>(xi + 4 * t);
        } else {
            for (int t = lane; t < d; t += 32)
                xs[t] = ldx(xi + t);
        }
        const int own = Lin[i];
        int u = collect_labels_plain(i, own, G, kappa, n, k, Lin, qlist, st);
        float bd = __int_as_float(0x7f800000);
        int br = 0x7fffffff;
        if constexpr (PART) {
            u = track_filter(trk, qlist, u);
            bd = best_out[i];
            br = own;
        }
        __syncwarp();
        // distances to the kept centroids, lane-parallel over candidates
        for (int q = lane; q < u; q += 32) {
            int r = qlist[q];
            float dv = cand_d2<VEC>(xs, C + (int64_t)r * d, d);
            if (key_less(dv, r, bd, br)) {
                bd = dv;
                br = r;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            float od = __shfl_xor_sync(FULL_MASK, bd, o);
            int orr = __shfl_xor_sync(FULL_MASK, br, o);
            if (key_less(od, orr, bd, br)) {
                bd = od;
                br = orr;
            }
        }
        write_winner(i, Lin, k, bd, br, Lout, best_out, trk);
        __syncwarp();
    });
}

// Coalesced variant for 16-byte rows (d % 4 == 0, d <= 32 * 4 * NV): the warp
// keeps x_i in registers (lane l owns vectors l, l + 32, ...; with LPR < 32 each
// set of LPR lanes holds the whole row and takes candidates of its own).  Distances are taken AS_G candidates at a
// time (AS_G / 2 for rows over 512 floats): each lane loads one 16-byte vector
// of every centroid of the group, and transpose_reduce completes the group's
// sums together.  The candidate list is padded to a multiple of the group with
// its first entry, whose second evaluation
// cannot change the (distance, label) minimum.
template <int NV, typename XT, int GS, bool LISTS, int LPR = 32>
__global__ void __launch_bounds__(AS_WARPS * 32, NV == 1 ? AS_ROWS_PER_SM : NV == 2 ? 5 : 4) k_assign_rows(
    const XT *__restrict__ X, int64_t n, int d, int64_t ld, const int32_t *__restrict__ G, int kappa,
    const float *__restrict__ C, int k, const int32_t *__restrict__ Lin, int32_t *__restrict__ Lout,
    float *__restrict__ best_out, DevStatus *st, const Track trk, const int32_t *__restrict__ todo)
{
    __shared__ __align__(16) int s_q[AS_WARPS][AS_QROW + (LPR < 32 ? GS * 32 / LPR : 0)];
    __shared__ __align__(16) int s_h[AS_WARPS][AS_HASH];
    const int w = threadIdx.x >> 5, lane = lane_id();
    int *qlist = s_q[w];
    int *tab = s_h[w];
    static_assert(GS == 4 || GS == 8, "candidates per lane set and group: 4 or 8");
    static_assert(LPR == 32 || (NV == 1 && LPR >= GS), "lane sets hold whole rows");
    constexpr int SETS = 32 / LPR;
    const int set = LPR == 32 ? 0 : lane / LPR, sl = LPR == 32 ? lane : lane % LPR;
    const int d4 = d >> 2;
    const float4 *C4 = reinterpret_cast<const float4 *>(C);

    each_sample<LISTS>((int64_t)blockIdx.x * AS_WARPS + w, (int64_t)gridDim.x * AS_WARPS, n, trk, todo,
                       [&](int64_t i, auto part_list) {
        constexpr bool PART = decltype(part_list)::value;
        const XT *xrow = X + i * ld;
        float4 xv[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) {
            int col = sl + 32 * v;
            xv[v] = col < d4 ? ldx4<XT, true>(xrow + 4 * col) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int own = Lin[i];
        int u = collect_labels<(LPR < 32)>(i, own, G, kappa, n, k, Lin, qlist, tab, st);
        float bd = __int_as_float(0x7f800000);
        int br = 0x7fffffff;
        if constexpr (PART) {
            u = track_filter(trk, qlist, u);
            bd = best_out[i];
            br = own;
        }
        if (u > 0 && lane < GS * SETS)
            qlist[u + lane] = qlist[0];
        __syncwarp();

        for (int g0 = 0; g0 < u; g0 += GS * SETS) {
            const int *ql = qlist + g0 + set * GS;
            int lab[GS];
#pragma unroll
            for (int c = 0; c < GS; c += 4) {
                const int4 q4 = *reinterpret_cast<const int4 *>(ql + c);
                lab[c] = q4.x;
                lab[c + 1] = q4.y;
                lab[c + 2] = q4.z;
                lab[c + 3] = q4.w;
            }
            float part[GS];
#pragma unroll
            for (int c = 0; c < GS; c++) {
                const float4 *row = C4 + (int64_t)lab[c] * d4;
                part[c] = lane_partial<NV, LPR>(xv, d4, [&](int col) { return __ldg(row + col); });
            }
            const float tot = transpose_reduce<GS, LPR>(part);
            const int r = ql[sl / (LPR / GS)];
            if (key_less(tot, r, bd, br)) {
                bd = tot;
                br = r;
            }
        }
        // lanes that share bits 4 .. log2(LPR / GS) hold the same candidates
#pragma unroll
        for (int o = 16; o >= LPR / GS; o >>= 1) {
            float od = __shfl_xor_sync(FULL_MASK, bd, o);
            int orr = __shfl_xor_sync(FULL_MASK, br, o);
            if (key_less(od, orr, bd, br)) {
                bd = od;
                br = orr;
            }
        }
        write_winner(i, Lin, k, bd, br, Lout, best_out, trk);
        __syncwarp();
    });
}

// k_assign_rows with the candidate distances screened against a BF16 shadow of
// the centroids (half the bytes per candidate row).  Pass 1 takes every
// candidate's distance D~ to the shadow row as k_assign_rows does (same lane
// layout, same candidate groups, shadow values widened exactly); with delta_r >=
// ||C_r - Cb_r||, |D - D~| <= delta_r (2 sqrt(D~) + delta_r) for the exact
// distances D, D~, and adding the FP32 rounding of both sums gives a bound E_r.
// Pass 2 recomputes, one at a time and against C, every candidate whose lower
// value D~ - E_r does not exceed the smallest upper value D~ + E_r (usually the
// winner alone), with the lane partials and summation tree of k_assign_rows,
// so the winner and its distance are that kernel's bit for bit.  The samples
// (FP32 or BF16, widened exactly) enter both passes unrounded: the bound covers
// the centroids' rounding alone.  SCR_TINY covers what the sums lose below
// FP32's normal range (at most 2^-150 a term); a bound that is no number keeps
// its candidate.
constexpr float SCR_TINY = 1e-41f;

template <int NV, typename XT, int GS, bool LISTS>
__global__ void __launch_bounds__(AS_WARPS * 32, NV <= 2 ? AS_ROWS_PER_SM : (NV == 4 ? 4 : 3)) k_assign_rows_scr(
    const XT *__restrict__ X, int64_t n, int d, int64_t ld, const int32_t *__restrict__ G, int kappa,
    const float *__restrict__ C, const void *__restrict__ Cs, const float *__restrict__ delta, int k,
    const int32_t *__restrict__ Lin, int32_t *__restrict__ Lout, float *__restrict__ best_out, DevStatus *st,
    const Track trk, const int32_t *__restrict__ todo)
{
    __shared__ __align__(16) int s_q[AS_WARPS][AS_QROW];
    __shared__ __align__(16) int s_h[AS_WARPS][AS_HASH];
    __shared__ float s_lo[AS_WARPS][AS_QROW];
    const int w = threadIdx.x >> 5, lane = lane_id();
    int *qlist = s_q[w];
    int *tab = s_h[w];
    float *lov = s_lo[w];
    static_assert(GS == 4 || GS == 8, "candidates per group: 4 or 8");
    const int d4 = d >> 2;
    const float4 *C4 = reinterpret_cast<const float4 *>(C);
    const uint2 *Cb4 = static_cast<const uint2 *>(Cs);  // 4 BF16 per 8 bytes
    const float gam = (float)(d + 8) * 5.9604645e-8f;         // FP32 rounding of a d-term sum, relative

    each_sample<LISTS>((int64_t)blockIdx.x * AS_WARPS + w, (int64_t)gridDim.x * AS_WARPS, n, trk, todo,
                       [&](int64_t i, auto part_list) {
        constexpr bool PART = decltype(part_list)::value;
        const XT *xrow = X + i * ld;
        float4 xv[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) {
            int col = lane + 32 * v;
            xv[v] = col < d4 ? ldx4<XT, true>(xrow + 4 * col) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int own = Lin[i];
        int u = collect_labels(i, own, G, kappa, n, k, Lin, qlist, tab, st);
        float bd = __int_as_float(0x7f800000);
        int br = 0x7fffffff;
        if constexpr (PART) {
            u = track_filter(trk, qlist, u);
            bd = best_out[i];
            br = own;
        }
        if (u > 0 && lane < GS)
            qlist[u + lane] = qlist[0];
        __syncwarp();

        // pass 1: BF16 distances with their bounds
        float best_up = bd;  // the known distance, or infinity
        for (int g0 = 0; g0 < u; g0 += GS) {
            int lab[GS];
#pragma unroll
            for (int c = 0; c < GS; c += 4) {
                const int4 q4 = *reinterpret_cast<const int4 *>(qlist + g0 + c);
                lab[c] = q4.x;
                lab[c + 1] = q4.y;
                lab[c + 2] = q4.z;
                lab[c + 3] = q4.w;
            }
            float part[GS];
#pragma unroll
            for (int c = 0; c < GS; c++) {
                const uint2 *row = Cb4 + (int64_t)lab[c] * d4;
                part[c] = lane_partial<NV>(xv, d4, [&](int col) { return bf16x4_to_float4(__ldg(row + col)); });
            }
            const float dt = transpose_reduce<GS>(part);
            const int cl = lane / (32 / GS);
            const float dl = __ldg(delta + qlist[g0 + cl]);
            const float sq = sqrtf(fmaxf(dt, 0.f));
            const float e = fmaf(1.01f, dl * (2.f * sq + dl) + gam * (2.f * dt + dl * (2.f * sq + dl)), SCR_TINY);
            if (lane % (32 / GS) == 0)
                lov[g0 + cl] = dt - e;
            best_up = fminf(best_up, dt + e);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            best_up = fminf(best_up, __shfl_xor_sync(FULL_MASK, best_up, o));
        __syncwarp();
        // pass 2: exact FP32 distances of the candidates that may be the minimum
        for (int g0 = 0; g0 < u; g0 += 32) {
            const int cnt = min(32, u - g0);
            unsigned sel = __ballot_sync(FULL_MASK, lane < cnt && !(lov[g0 + lane] > best_up));
            while (sel) {
                const int c = __ffs(sel) - 1;
                sel &= sel - 1;
                const int r = qlist[g0 + c];
                const float4 *row = C4 + (int64_t)r * d4;
                const float tot = warp_total(lane_partial<NV>(xv, d4, [&](int col) { return __ldg(row + col); }));
                if (key_less(tot, r, bd, br)) {
                    bd = tot;
                    br = r;
                }
            }
        }
        write_winner(i, Lin, k, bd, br, Lout, best_out, trk);
        __syncwarp();
    });
}

// ---------------------------------------------------------------------------
// BF16 shadow of the centroids: Cb = bf16(C) and delta_r >= ||C_r - Cb_r||.
// ---------------------------------------------------------------------------
__global__ void k_shadow_bf16(const float *__restrict__ C, int k, int d, __nv_bfloat16 *__restrict__ Cb,
                              float *__restrict__ delta, float *__restrict__ cnorm, const uint8_t *__restrict__ dirty)
{
    const int lane = lane_id();
    for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < k; r += gridDim.x * (blockDim.x >> 5)) {
        if (dirty && dirty[r] == 0)
            continue;  // the row, and so its shadow, is as the previous assignment left it
        double e = 0.0, c2 = 0.0;
        for (int t = lane; t < d; t += 32) {
            const float c = C[(int64_t)r * d + t];
            const __nv_bfloat16 b = __float2bfloat16_rn(c);
            Cb[(int64_t)r * d + t] = b;
            const double diff = (double)c - (double)__bfloat162float(b);
            e += diff * diff;
            c2 += (double)c * (double)c;
        }
        for (int o = 16; o > 0; o >>= 1) {
            e += __shfl_xor_sync(FULL_MASK, e, o);
            c2 += __shfl_xor_sync(FULL_MASK, c2, o);
        }
        if (lane == 0) {
            delta[r] = (float)(sqrt(e) * (1.0 + 1e-6)) + 1e-30f;  // rounded up
            cnorm[r] = (float)c2;                                 // ||C_r||^2 (a bound input only)
        }
    }
}

// Int8 shadow of the centroids: per row r the scale s_r = max_t |C_rt| / 127 (1 for a zero row), codes
// q_rt = rint(C_rt / s_r) (the quotient taken as a product with 1 / s_r) in [-127, 127], coordinate t at byte t of a
// row of 16 * units bytes (zeros past d), and meta[r] = {s_r, s_r^2 sum q^2, delta_r, 0} with
// delta_r >= ||C_r - q_r s_r||, in FP32
// only.  Each error v - q s is formed as (v - p) - e with p = fl(q s) and e = fma(q, s, -p) (q s = p + e
// exactly); v - p is exact where p/2 <= v <= 2p (Sterbenz; |q| >= 1 puts v within half a step of q s), so the
// computed error is within 2u |v - q s| + 1.01 u^2 max|C_r| of the true one (u = 2^-24).  The errors are squared
// in units of w = max(s, FLT_MIN) (so that no square of a row of tiny values falls below the normal range) and
// summed in FP32 (d fma steps and the warp's 5 additions: relative error below gamma_(d+5), one more u for the
// division by w); delta_r inflates the square root by (d + 24) 1.2e-7 and 1e-5 (the 1 / (1 - 2u) above and this
// evaluation's own roundings) and adds sqrt(d) 4e-15 max|C_r| (the absolute term, which also covers squares
// below the normal range): a rigorous upper bound, no FP64.  sum q^2 <= 1024 * 127^2 is exact in FP32.  A row that is
// not finite has zero codes and an infinite delta_r (always recomputed).
__global__ void k_shadow_i8(const float *__restrict__ C, int k, int d, int units, uint32_t *__restrict__ Cq,
                            float4 *__restrict__ meta, const uint8_t *__restrict__ dirty)
{
    const int lane = lane_id();
    const int d4 = d >> 2, words = units * 4;
    for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < k; r += gridDim.x * (blockDim.x >> 5)) {
        if (dirty && dirty[r] == 0)
            continue;  // the row, and so its shadow, is as the previous assignment left it
        const float4 *row = reinterpret_cast<const float4 *>(C + (int64_t)r * d);
        unsigned mb = 0;  // the largest magnitude's bits (in order; infinities and NaN above every number)
        for (int col = lane; col < d4; col += 32) {
            const float4 v = row[col];
            mb = max(max(mb, __float_as_uint(fabsf(v.x))), __float_as_uint(fabsf(v.y)));
            mb = max(max(mb, __float_as_uint(fabsf(v.z))), __float_as_uint(fabsf(v.w)));
        }
        mb = __reduce_max_sync(FULL_MASK, mb);
        const bool finite = mb < 0x7f800000u;
        const float mx = finite ? __uint_as_float(mb) : 0.f;
        const float sc = mx > 0.f ? mx / 127.f : 1.f;
        const float inv = 1.f / sc;
        const float wu = fmaxf(sc, 1.17549435e-38f), winv = 1.f / wu;  // error unit (FLT_MIN at least)
        float e = 0.f;
        int qq = 0;
        for (int col = lane; col < words; col += 32) {
            uint32_t word = 0;
            if (finite && col < d4) {
                const float4 v = row[col];
                const float vals[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const float qf = fminf(127.f, fmaxf(-127.f, rintf(vals[q] * inv)));
                    const int qi = (int)qf;
                    word |= (uint32_t)(qi & 0xff) << (8 * q);
                    qq += qi * qi;
                    const float p = qf * sc;
                    const float pe = fmaf(qf, sc, -p);  // q s = p + pe exactly
                    const float z = ((vals[q] - p) - pe) * winv;
                    e = fmaf(z, z, e);
                }
            }
            Cq[(int64_t)r * words + col] = word;
        }
        for (int o = 16; o > 0; o >>= 1)
            e += __shfl_xor_sync(FULL_MASK, e, o);
        qq = __reduce_add_sync(FULL_MASK, qq);
        if (lane == 0) {
            const float delta = sqrtf(e * (1.f + (float)(d + 24) * 1.2e-7f)) * 1.00001f * wu +
                                sqrtf((float)d) * 4e-15f * mx + 1e-30f;
            meta[r] = finite ? make_float4(sc, sc * sc * (float)qq, delta, 0.f)
                             : make_float4(0.f, 0.f, __int_as_float(0x7f800000), 0.f);
        }
    }
}

// Four signed bytes by four, added to c.
__device__ __forceinline__ int dot4(uint32_t a, uint32_t b, int c) { return __dp4a((int)a, (int)b, c); }

// k_assign_rows with the candidates screened against the int8 shadow in integer arithmetic.  The sample is coded in 15
// bits, x_t = s_x (128 h_t + l_t) + error with s_x = max|x| / 16256 and signed bytes h, l, so that a candidate's
// product with it is exact in two __dp4a per four coordinates, where widening the codes to FP32 took ten instructions
// (and bounded this pass: 75 warp instructions a candidate at d = 512, about 20 now).  A row of the shadow is 16 * LPR *
// NW bytes (the smallest that hold d): LPR lanes read one candidate's row, 16 bytes each, NW times, so a warp takes 32 /
// LPR candidates at once.  With X2 = |x~|^2 and C2 = |c~|^2 of the coded vectors,
//   D~ = X2 + C2 - 2 s_x s_r dot,
// the true distance's root is within delta = delta_r + 0.51 s_x sqrt(d) of the coded one's; to
// E = delta (2 sqrt(D~ + er) + delta) come er = 64 2^-24 (X2 + C2) + 2^-117 for the FP32 evaluation of D~ (X2 summed over
// at most 32 terms a lane and 5 steps; below FP32's normal range s_x s_r is off by up to 2^-150, times |dot| < 2^31, and
// the other products and the canonical sum by less) and the rounding gam of the canonical sum.  Pass 2 recomputes every
// candidate whose lower value does not exceed the smallest upper value, as the BF16 form does, with the same bits.  A
// sample that is not finite, or with at most Q8_FEW candidates, goes to pass 2 whole.
constexpr int Q8_FEW = 3;

template <int LPR, int NW, int NV, typename XT, bool LISTS>
__global__ void __launch_bounds__(AS_WARPS * 32, NV <= 2 ? AS_ROWS_PER_SM : 4) k_assign_rows_scr(
    const XT *__restrict__ X, int64_t n, int d, int64_t ld, const int32_t *__restrict__ G, int kappa,
    const float *__restrict__ C, const uint4 *__restrict__ Cq, const float4 *__restrict__ meta, int k,
    const int32_t *__restrict__ Lin, int32_t *__restrict__ Lout, float *__restrict__ best_out, DevStatus *st,
    const Track trk, const int32_t *__restrict__ todo)
{
    __shared__ __align__(16) int s_q[AS_WARPS][AS_QROW];
    __shared__ __align__(16) int s_h[AS_WARPS][AS_HASH];
    __shared__ float s_lo[AS_WARPS][AS_QROW];
    const int w = threadIdx.x >> 5, lane = lane_id();
    int *qlist = s_q[w];
    int *tab = s_h[w];
    float *lov = s_lo[w];
    constexpr int G4 = 32 / LPR;                  // candidates side by side
    constexpr int U = LPR == 32 ? 4 : LPR == 16 ? 2 : 1;  // such groups in flight (LPR = 32: a transposed reduction)
    const int sub = lane % LPR, grp = lane / LPR;
    const int d4 = d >> 2;
    const float4 *C4 = reinterpret_cast<const float4 *>(C);
    const float gam = (float)(d + 8) * 5.9604645e-8f;  // FP32 rounding of a d-term sum, relative
    const float rootd = 0.51f * sqrtf((float)d);

    each_sample<LISTS>((int64_t)blockIdx.x * AS_WARPS + w, (int64_t)gridDim.x * AS_WARPS, n, trk, todo,
                       [&](int64_t i, auto part_list) {
        constexpr bool PART = decltype(part_list)::value;
        const XT *xrow = X + i * ld;
        // this lane's 16 coordinates of every 16 * LPR
        float4 v[NW * 4];
#pragma unroll
        for (int q = 0; q < NW * 4; q++) {
            const int col = ((q >> 2) * LPR + sub) * 4 + (q & 3);
            v[q] = col < d4 ? ldx4<XT>(xrow + 4 * col) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int own = Lin[i];
        int u = collect_labels(i, own, G, kappa, n, k, Lin, qlist, tab, st);
        float bd = __int_as_float(0x7f800000);
        int br = 0x7fffffff;
        if constexpr (PART) {
            u = track_filter(trk, qlist, u);
            bd = best_out[i];
            br = own;
        }
        unsigned mb = 0;
#pragma unroll
        for (int q = 0; q < NW * 4; q++) {
            mb = max(max(mb, __float_as_uint(fabsf(v[q].x))), __float_as_uint(fabsf(v[q].y)));
            mb = max(max(mb, __float_as_uint(fabsf(v[q].z))), __float_as_uint(fabsf(v[q].w)));
        }
        mb = __reduce_max_sync(FULL_MASK, mb);
        const bool screen = u > Q8_FEW && mb < 0x7f800000u;
        float best_up = bd;  // the known distance, or infinity
        if (screen) {
            if (lane < G4 * U)
                qlist[u + lane] = qlist[0];
            __syncwarp();
            const float mx = fmaxf(__uint_as_float(mb), 1e-30f);
            const float sx = mx / 16256.f, inv = 16256.f / mx;
            uint32_t hx[NW * 4], lx[NW * 4];
            float x2 = 0.f;
#pragma unroll
            for (int q = 0; q < NW * 4; q++) {
                const float vals[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
                uint32_t hw = 0, lw = 0;
#pragma unroll
                for (int z = 0; z < 4; z++) {
                    // rint(x / s_x) in the low bits of a float (magnitude below 2^22)
                    const float t = fmaf(vals[z], inv, 12582912.f);
                    const int c = __float_as_int(t) - 0x4b400000, h = (c + 64) >> 7;
                    const float f = t - 12582912.f;
                    x2 = fmaf(f, f, x2);
                    hw |= (uint32_t)(h & 0xff) << (8 * z);
                    lw |= (uint32_t)((c - (h << 7)) & 0xff) << (8 * z);
                }
                hx[q] = hw;
                lx[q] = lw;
            }
#pragma unroll
            for (int o = LPR / 2; o > 0; o >>= 1)
                x2 += __shfl_xor_sync(FULL_MASK, x2, o);
            const float X2 = x2 * sx * sx, dx = rootd * sx;
            // candidate c's lower and upper values, from its dot product with the sample
            auto bounds = [&](int c, int dot, bool first) {
                const float4 mt = __ldg(meta + qlist[c]);
                const float n2 = X2 + mt.y;
                const float dt = fmaf(-2.f * sx * mt.x, (float)dot, n2);
                const float er = fmaf(3.8146973e-6f, n2, 6.0e-36f), dl = mt.z + dx;
                const float dp = fmaxf(dt, 0.f) + er;
                const float sq = dl * (2.f * sqrtf(dp) + dl);
                const float e = 1.01f * (sq + er + gam * (2.f * dp + sq));
                float lo = dt - e, up = dt + e;
                if (!(fabsf(dt) < 1e37f) || !(e < 1e37f))
                    lo = -__int_as_float(0x7f800000), up = __int_as_float(0x7f800000);
                if (first)
                    lov[c] = lo;
                best_up = fminf(best_up, up);
            };
            for (int c0 = 0; c0 < u; c0 += G4 * U) {
                int part[U];
#pragma unroll
                for (int z = 0; z < U; z++) {
                    const uint4 *row = Cq + (int64_t)qlist[c0 + z * G4 + grp] * (LPR * NW) + sub;
                    int hh = 0, ll = 0;
#pragma unroll
                    for (int q = 0; q < NW; q++) {
                        const uint4 cw = __ldg(row + q * LPR);
                        hh = dot4(cw.x, hx[4 * q], hh);
                        hh = dot4(cw.y, hx[4 * q + 1], hh);
                        hh = dot4(cw.z, hx[4 * q + 2], hh);
                        hh = dot4(cw.w, hx[4 * q + 3], hh);
                        ll = dot4(cw.x, lx[4 * q], ll);
                        ll = dot4(cw.y, lx[4 * q + 1], ll);
                        ll = dot4(cw.z, lx[4 * q + 2], ll);
                        ll = dot4(cw.w, lx[4 * q + 3], ll);
                    }
                    part[z] = (hh << 7) + ll;  // |sum over d <= 1024| < 2^31
                }
                if constexpr (LPR == 32) {
                    // four sums at once: lane l ends with candidate l / 8
                    const bool up = (lane & 16) != 0, up2 = (lane & 8) != 0;
                    int a = (up ? part[2] : part[0]) + __shfl_xor_sync(FULL_MASK, up ? part[0] : part[2], 16);
                    const int b = (up ? part[3] : part[1]) + __shfl_xor_sync(FULL_MASK, up ? part[1] : part[3], 16);
                    a = (up2 ? b : a) + __shfl_xor_sync(FULL_MASK, up2 ? a : b, 8);
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1)
                        a += __shfl_xor_sync(FULL_MASK, a, o);
                    bounds(c0 + (lane >> 3), a, (lane & 7) == 0);
                } else {
#pragma unroll
                    for (int z = 0; z < U; z++) {
#pragma unroll
                        for (int o = LPR / 2; o > 0; o >>= 1)
                            part[z] += __shfl_xor_sync(FULL_MASK, part[z], o);
                        bounds(c0 + z * G4 + grp, part[z], sub == 0);
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                best_up = fminf(best_up, __shfl_xor_sync(FULL_MASK, best_up, o));
        }
        __syncwarp();
        // pass 2: exact FP32 distances of the candidates that may be the minimum
        float4 xv[NV];
#pragma unroll
        for (int q = 0; q < NV; q++) {
            const int col = lane + 32 * q;
            xv[q] = col < d4 ? ldx4<XT>(xrow + 4 * col) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int g0 = 0; g0 < u; g0 += 32) {
            const int cnt = min(32, u - g0);
            unsigned sel = __ballot_sync(FULL_MASK, lane < cnt && (!screen || lov[g0 + lane] <= best_up));
            while (sel) {
                const int c = __ffs(sel) - 1;
                sel &= sel - 1;
                const int r = qlist[g0 + c];
                const float4 *row = C4 + (int64_t)r * d4;
                const float tot = warp_total(lane_partial<NV>(xv, d4, [&](int col) { return __ldg(row + col); }));
                if (key_less(tot, r, bd, br)) {
                    bd = tot;
                    br = r;
                }
            }
        }
        write_winner(i, Lin, k, bd, br, Lout, best_out, trk);
        __syncwarp();
    });
}

// k_assign_rows with the candidate distances first taken against the BF16
// shadow Cb (half the bytes per candidate row).  With delta_r >= ||C_r - Cb_r||,
// |D - D~| <= delta_r (2 sqrt(D~) + delta_r) for the exact distances D, D~ to
// C_r and Cb_r; adding the FP32 rounding of both sums gives a bound E_r, and
// every candidate whose lower value D~ - E_r does not exceed the smallest upper
// value D~ + E_r is recomputed against C with the FP32 kernel's order (same
// lane partials, same reduction tree), so the winner and its distance are the
// FP32 kernel's bit for bit.
template <int NV, bool TILES>
__global__ void __launch_bounds__(AS_WARPS * 32) k_assign_rows_bf(const float *__restrict__ X, int64_t n, int d,
                                                                  int64_t ld, const int32_t *__restrict__ G,
                                                                  int kappa, const float *__restrict__ C,
                                                                  const __nv_bfloat16 *__restrict__ Cb,
                                                                  const float *__restrict__ delta, int k,
                                                                  const int32_t *__restrict__ Lin,
                                                                  int32_t *__restrict__ Lout,
                                                                  float *__restrict__ best_out,
                                                                  const int32_t *__restrict__ tmem_members,
                                                                  const int32_t *__restrict__ tile_flag,
                                                                  const int32_t *__restrict__ sel_lab,
                                                                  const int32_t *__restrict__ sel_n, DevStatus *st,
                                                                  unsigned *__restrict__ ticket)
{
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *ticket = 0u;  // for k_assign_reduce
    __shared__ int s_q[AS_WARPS][AS_QCAP];
    __shared__ float s_lo[AS_WARPS][AS_QCAP + 31];
    const int w = threadIdx.x >> 5, lane = lane_id();
    int *qlist = s_q[w];
    const int d4 = d >> 2;
    const float4 *C4 = reinterpret_cast<const float4 *>(C);
    const uint2 *Cb4 = reinterpret_cast<const uint2 *>(Cb);  // 4 BF16 per 8 bytes
    const float gam = (float)(d + 8) * 5.9604645e-8f;         // FP32 rounding of a d-term sum, relative

    const int ncand = kappa + 1;
    for (int64_t p = (int64_t)blockIdx.x * AS_WARPS + w; p < n; p += (int64_t)gridDim.x * AS_WARPS) {
        int64_t i = p;
        int nl = -1;  // >= 0: the tensor-core screening left nl candidates for the exact pass
        if (TILES) {
            i = tmem_members[p];
            if (!tile_flag[p / AS_TILE])
                nl = sel_n[i];
        }
        const float4 *x4 = reinterpret_cast<const float4 *>(X + i * ld);
        float4 xv[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) {
            int col = lane + 32 * v;
            xv[v] = col < d4 ? __ldcs(x4 + col) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int own = Lin[i];
        float bd = __int_as_float(0x7f800000);
        int br = 0x7fffffff;
        if (nl >= 0) {
            // exact FP32 distances of the screened labels (same lane partials and reduction grouping)
            const int mine = lane < nl ? __ldg(sel_lab + i * 8 + lane) : 0;
#pragma unroll 4
            for (int z = 0; z < nl; z++) {
                const int r = __shfl_sync(FULL_MASK, mine, z);
                const float4 *row = C4 + (int64_t)r * d4;
                const float tot = warp_total(lane_partial<NV>(xv, d4, [&](int col) { return __ldg(row + col); }));
                if (key_less(tot, r, bd, br)) {
                    bd = tot;
                    br = r;
                }
            }
        } else {
            int u = 0;
            for (int c0 = 0; c0 < ncand; c0 += 32) {
                int c = c0 + lane;
                int lab = -1;
                if (c == 0) {
                    lab = own;
                } else if (c < ncand) {
                    int nb = __ldcs(G + i * kappa + (c - 1));
                    if ((unsigned)nb < (unsigned)n)
                        lab = Lin[nb];
                    else
                        flag_error(st, GK_ERR_INVALID, (unsigned)i);
                }
                if (c < ncand && (unsigned)lab >= (unsigned)k) {
                    flag_error(st, GK_ERR_INVALID, (unsigned)i);
                    lab = -1;
                }
                unsigned peers = __match_any_sync(FULL_MASK, lab);
                bool keep = lab >= 0 && (peers & lanemask_lt()) == 0u;
                if (keep)
                    for (int q = 0; q < u; q++)
                        if (qlist[q] == lab) {
                            keep = false;
                            break;
                        }
                unsigned keeps = __ballot_sync(FULL_MASK, keep);
                __syncwarp();
                if (keep)
                    qlist[u + __popc(keeps & lanemask_lt())] = lab;
                u += __popc(keeps);
                __syncwarp();
            }
            // pass 1: BF16 distances of every candidate (lane l holds candidate g0 + l of each group)
            float *lov = s_lo[w];
            float best_up = __int_as_float(0x7f800000);
#pragma unroll 1
            for (int g0 = 0; g0 < u; g0 += 32) {
                const int cnt = min(32, u - g0);
                float part[32];
#pragma unroll
                for (int c = 0; c < 32; c++) {
                    float acc = 0.f;
                    if (c < cnt) {
                        const uint2 *row = Cb4 + (int64_t)qlist[g0 + c] * d4;
                        acc = lane_partial<NV>(xv, d4, [&](int col) { return bf16x4_to_float4(__ldg(row + col)); });
                    }
                    part[c] = acc;
                }
                const float dt = transpose_reduce32(part);
                if (lane < cnt) {
                    const float dl = delta[qlist[g0 + lane]];
                    const float sq = sqrtf(fmaxf(dt, 0.f));
                    const float e =
                        fmaf(1.01f, dl * (2.f * sq + dl) + gam * (2.f * dt + dl * (2.f * sq + dl)), SCR_TINY);
                    lov[g0 + lane] = dt - e;
                    best_up = fminf(best_up, dt + e);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                best_up = fminf(best_up, __shfl_xor_sync(FULL_MASK, best_up, o));
            __syncwarp();
            // pass 2: FP32 distances of the candidates that may be the minimum, one at a
            // time; the xor butterfly groups the lane partials as transpose_reduce32 does,
            // so each total has the bits of the FP32 kernel
#pragma unroll 1
            for (int g0 = 0; g0 < u; g0 += 32) {
                const int cnt = min(32, u - g0);
                unsigned sel = __ballot_sync(FULL_MASK, lane < cnt && !(lov[g0 + lane] > best_up));
                while (sel) {
                    const int c = __ffs(sel) - 1;
                    sel &= sel - 1;
                    const int r = qlist[g0 + c];
                    const float4 *row = C4 + (int64_t)r * d4;
                    float tot = lane_partial<NV>(xv, d4, [&](int col) { return __ldg(row + col); });
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        tot += __shfl_xor_sync(FULL_MASK, tot, o);
                    if (key_less(tot, r, bd, br)) {
                        bd = tot;
                        br = r;
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            float od = __shfl_xor_sync(FULL_MASK, bd, o);
            int orr = __shfl_xor_sync(FULL_MASK, br, o);
            if (key_less(od, orr, bd, br)) {
                bd = od;
                br = orr;
            }
        }
        if (lane == 0) {
            if (br == 0x7fffffff)  // no valid candidate (own label out of range): keep the input label
                br = own, bd = 0.f;
            Lout[i] = br;
            if (best_out)
                best_out[i] = bd;
        }
        __syncwarp();
    }
}

// FP64 sum of best[] and count of changed labels: per block over fixed index ranges (the same for every kernel that
// produced best[], so the total has the same bits whichever assignment kernel ran), then over the blocks in the order
// of 1024 chains and a halving tree, by the last block to finish (trk.ticket; a launch of its own took 3.6 us and a
// gap).
__global__ void __launch_bounds__(256) k_assign_reduce(const float *__restrict__ best,
                                                       const int32_t *__restrict__ Lin,
                                                       const int32_t *__restrict__ Lout, int64_t n,
                                                       double *__restrict__ blk_sum,
                                                       unsigned long long *__restrict__ blk_changed, const Track trk,
                                                       int k, double *__restrict__ sum_d2,
                                                       int64_t *__restrict__ n_changed)
{
    static_assert(AS_BLOCKS > 1024 && AS_BLOCKS <= 2048, "two blocks per chain at most");
    if (trk.dirty_out)  // for the next assignment's k_assign_select
        for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
            const int r = Lout[i];
            trk.mark[i] = (unsigned)r < (unsigned)k ? trk.dirty_out[r] : 1;
        }
    if (trk.clear) {  // Track's clears, here to save a launch
        for (int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x; r < k; r += (int64_t)gridDim.x * 256)
            trk.clear[r] = 0;
        if (blockIdx.x == 0 && threadIdx.x < 2)
            trk.todo_n[threadIdx.x] = 0;
    }
    __shared__ double s[1024];
    __shared__ unsigned long long c[1024];
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = min(n, b0 + per);
    double a = 0.0;
    unsigned long long ch = 0;
    for (int64_t i = b0 + threadIdx.x; i < b1; i += 256) {
        a += (double)best[i];
        ch += Lin[i] != Lout[i] ? 1ull : 0ull;
    }
    s[threadIdx.x] = a;
    c[threadIdx.x] = ch;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            s[threadIdx.x] += s[threadIdx.x + o];
            c[threadIdx.x] += c[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        blk_sum[blockIdx.x] = s[0];
        blk_changed[blockIdx.x] = c[0];
    }
    if (!last_block(trk.ticket))
        return;
    for (int q = threadIdx.x; q < 1024; q += 256) {
        double x = __ldcg(blk_sum + q);
        unsigned long long y = __ldcg(blk_changed + q);
        if (q + 1024 < (int)gridDim.x) {
            x += __ldcg(blk_sum + q + 1024);
            y += __ldcg(blk_changed + q + 1024);
        }
        s[q] = x;
        c[q] = y;
    }
    __syncthreads();
    halving_sum<256>(s, 1024);
    halving_sum<256>(c, 1024);
    if (threadIdx.x == 0) {
        if (sum_d2)
            *sum_d2 = s[0];
        if (n_changed)
            *n_changed = (int64_t)c[0];
    }
}

static size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

size_t assign_scratch_bytes(int64_t n, int32_t k, int64_t d)
{
    const size_t part = al256((size_t)AS_BLOCKS * (sizeof(double) + sizeof(unsigned long long)) + sizeof(unsigned));
    const size_t shadow = al256((size_t)k * (size_t)d * 2) + 2 * al256((size_t)k * 4) + al256((size_t)k * 16);
    const size_t best = al256((size_t)n * 4);
    const size_t tiles = al256((size_t)((n + AS_TILE - 1) / AS_TILE) * 4);
    const size_t sel = al256((size_t)n * 8 * 4) + al256((size_t)n * 4);
    return part + shadow + best + tiles + sel;
}

// Narrowest rows the int8 screening takes (a row of the shadow has at least 64 bytes, in the place of 2 d).
constexpr int Q8_MIN_D = 32;

// 16-byte vectors of a row of the int8 shadow.
static int q8_units(int64_t d) { return d <= 64 ? 4 : d <= 128 ? 8 : d <= 256 ? 16 : d <= 512 ? 32 : 64; }

// Where precision 1 takes the int8 screening (0 never does): rows of more than Q8_PAYS_D values, where the bytes that a
// sample's candidates spare, min(kappa, k) times a row's, outweigh what the screening costs a sample (its bounds, the
// shadow's k / n rows, its launch); not for few clusters, whose samples have few distinct candidates.  FP32 rows against
// screening, us an assignment in the middle of a fit:
//   200k x 256, k = 2k, kappa = 20  230 / 300     300k x 128, k = 3k, kappa = 20 401 / 516    (Q8_PAYS_D)
//   100k x 300, k = 2k, kappa = 20  200 / 183     kappa = 10  151 / 154     k = n, kappa = 20 239 / 255
//   200k x 512 BF16, k = 4k, kappa = 20  457 / 349     kappa = 10  306 / 280     kappa = 4  206 / 241
//   100k x 960, k = 2k, kappa = 10  390 / 258     k = n, kappa = 50  2947 / 702     k = 10, kappa = 50  263 / 305
//   15k x 300, k = 300, kappa = 20  62 / 63       9k x 512, k = 900, kappa = 10  52 / 57     (2^22 values or few more)
constexpr int Q8_PAYS_D = 288;
constexpr int Q8_PAYS_K = 100;

static bool assign_q8_pays(int64_t n, int64_t d, int32_t k, int32_t kappa)
{
    const int64_t large = (int64_t)1 << 22;
    if (d <= Q8_PAYS_D || n * d < large || k < Q8_PAYS_K)
        return false;
    const int64_t spared = std::min(kappa, k) * (4 * d - 16 * q8_units(d));
    return spared >= 12000 + 3000 * (int64_t)k / n + 8000 * large / (n * d);
}

template <typename XT>
static cudaError_t assign_t(const XT *X, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx, int32_t kappa,
                            const float *C, int32_t k, const int32_t *labels_in, int32_t *labels_out, float *best_d2,
                            double *sum_d2, int64_t *n_changed, void *scratch, DevStatus *st, cudaStream_t s,
                            int precision, const int32_t *members, Track trk)
{
    char *sp = static_cast<char *>(scratch);
    double *blk_sum = reinterpret_cast<double *>(sp);
    unsigned long long *blk_chg = reinterpret_cast<unsigned long long *>(blk_sum + AS_BLOCKS);
    trk.ticket = reinterpret_cast<unsigned *>(blk_chg + AS_BLOCKS);
    sp += al256((size_t)AS_BLOCKS * (sizeof(double) + sizeof(unsigned long long)) + sizeof(unsigned));
    __nv_bfloat16 *Cb = reinterpret_cast<__nv_bfloat16 *>(sp);
    sp += al256((size_t)k * (size_t)d * 2);
    float *delta = reinterpret_cast<float *>(sp);
    sp += al256((size_t)k * 4);
    float *cnorm = reinterpret_cast<float *>(sp);
    sp += al256((size_t)k * 4);
    float4 *meta = reinterpret_cast<float4 *>(sp);
    sp += al256((size_t)k * 16);
    float *best = best_d2 ? best_d2 : reinterpret_cast<float *>(sp);
    sp += al256((size_t)n * 4);
    int32_t *tile_flag = reinterpret_cast<int32_t *>(sp);
    sp += al256((size_t)((n + AS_TILE - 1) / AS_TILE) * 4);
    int32_t *sel_lab = reinterpret_cast<int32_t *>(sp);
    sp += al256((size_t)n * 8 * 4);
    int32_t *sel_n = reinterpret_cast<int32_t *>(sp);

    const bool vec4 = x_vec4(X, d, ld) && ((reinterpret_cast<uintptr_t>(C) & 15) == 0);
    const int d4 = (int)(d / 4);
    // candidates per group of the row kernels (a tile shape: every width gives the same bits, transpose_reduce
    // forms each total with warp_total's tree): 8 by default, 4 for rows of more than 512 values, where 8 would
    // not keep the loads in registers; a caller (the autotuner) may ask for 4 or 8.  Rows of at most 64 (32) values
    // of precision 0 and 1 take two (four) candidates to a load, four loads a group: 1.3M x 64, kappa = 20 329 us
    // an assignment instead of 422 (eight loads a group 392); 20k x 32 9.1 us instead of 11.6 (eight 11.0)
    const int gw = (precision >> 8) & 0xff;
    precision &= 0xff;
    cudaError_t e;
    int grid = 0;
    bool done = false;
    if (trk.dirty) {  // the lists take the place that precision 3 alone uses otherwise
        const int64_t sb = (n + SL_WARPS * 32 - 1) / (SL_WARPS * 32);
        const unsigned sgrid = (unsigned)(sb < 152 * 8 ? sb : 152 * 8);
        if (kappa <= 32)
            k_assign_select<1><<<sgrid, SL_WARPS * 32, 0, s>>>(n, g_idx, kappa, k, labels_in, labels_out, trk, sel_lab);
        else if (kappa <= 64)
            k_assign_select<2><<<sgrid, SL_WARPS * 32, 0, s>>>(n, g_idx, kappa, k, labels_in, labels_out, trk, sel_lab);
        else
            k_assign_select<4><<<sgrid, SL_WARPS * 32, 0, s>>>(n, g_idx, kappa, k, labels_in, labels_out, trk, sel_lab);
    }
    // The int8 screening at precision 4, and at 1 where it is faster than the FP32 rows (assign_q8_pays): the results
    // are the same.
    const bool q8 = vec4 && d >= Q8_MIN_D && d4 <= 32 * 8 &&
                    (precision == 4 || (precision == 1 && assign_q8_pays(n, d, k, kappa)));
    if (q8) {
        const int sgrid = (k + 7) / 8 < 152 * 16 ? (k + 7) / 8 : 152 * 16;
        k_shadow_i8<<<sgrid, 256, 0, s>>>(C, k, (int)d, q8_units(d), reinterpret_cast<uint32_t *>(Cb), meta, trk.dirty);
        auto launch = [&](auto kernel) -> cudaError_t {
            cudaError_t le = resident_grid(reinterpret_cast<const void *>(kernel), AS_WARPS * 32, 0, &grid);
            if (le == cudaSuccess)
                kernel<<<grid, AS_WARPS * 32, 0, s>>>(X, n, (int)d, ld, g_idx, kappa, C, reinterpret_cast<const uint4 *>(Cb),
                                                      meta, k, labels_in, labels_out, best, st, trk, sel_lab);
            return le;
        };
#define GK_ASQ8(LPR, NW, NV) \
    (trk.dirty ? launch(k_assign_rows_scr<LPR, NW, NV, XT, true>) : launch(k_assign_rows_scr<LPR, NW, NV, XT, false>))
        e = d <= 64    ? GK_ASQ8(4, 1, 1)
            : d <= 128 ? GK_ASQ8(8, 1, 1)
            : d <= 256 ? GK_ASQ8(16, 1, 2)
            : d <= 512 ? GK_ASQ8(32, 1, 4)
                       : GK_ASQ8(32, 2, 8);
#undef GK_ASQ8
        if (e != cudaSuccess)
            return e;
        done = true;
    } else if (precision == 2 && vec4 && d4 <= 32 * 8) {
        const int sgrid = (k + 7) / 8 < 152 * 16 ? (k + 7) / 8 : 152 * 16;
        k_shadow_bf16<<<sgrid, 256, 0, s>>>(C, k, (int)d, Cb, delta, cnorm, trk.dirty);
        auto launch = [&](auto kernel) -> cudaError_t {
            cudaError_t le = resident_grid(reinterpret_cast<const void *>(kernel), AS_WARPS * 32, 0, &grid);
            if (le == cudaSuccess)
                kernel<<<grid, AS_WARPS * 32, 0, s>>>(X, n, (int)d, ld, g_idx, kappa, C, Cb, delta, k, labels_in, labels_out,
                                                      best, st, trk, sel_lab);
            return le;
        };
#define GK_ASBF(NV, GS) \
    (trk.dirty ? launch(k_assign_rows_scr<NV, XT, GS, true>) : launch(k_assign_rows_scr<NV, XT, GS, false>))
        if (d4 <= 32)
            e = gw == 4 ? GK_ASBF(1, 4) : GK_ASBF(1, 8);
        else if (d4 <= 64)
            e = gw == 4 ? GK_ASBF(2, 4) : GK_ASBF(2, 8);
        else if (d4 <= 128)
            e = gw == 4 ? GK_ASBF(4, 4) : GK_ASBF(4, 8);
        else
            e = GK_ASBF(8, 4);
#undef GK_ASBF
        if (e != cudaSuccess)
            return e;
        done = true;
    }
    if constexpr (std::is_same_v<XT, float>) {  // tensor-core screening: FP32 samples only
        if (precision == 3 && vec4 && d4 <= 32 * 8) {
            k_shadow_bf16<<<(k + 7) / 8 < 152 * 16 ? (k + 7) / 8 : 152 * 16, 256, 0, s>>>(C, k, (int)d, Cb, delta,
                                                                                      cnorm, nullptr);
            const bool tiles = members && assign_tc_supported(d, ld, X, C, kappa);
            if (tiles) {
                if ((e = launch_assign_tc(X, n, d, ld, g_idx, kappa, C, Cb, delta, cnorm, k, labels_in, members,
                                          sel_lab, sel_n, tile_flag, st, s)) != cudaSuccess)
                    return e;
            }
#define GK_ASGB(NV, T)                                                                                           \
    k_assign_rows_bf<NV, T><<<AS_BLOCKS, AS_WARPS * 32, 0, s>>>(X, n, (int)d, ld, g_idx, kappa, C, Cb, delta, k,   \
                                                                labels_in, labels_out, best,                        \
                                                                members, tile_flag, sel_lab, sel_n, st, trk.ticket)
            if (tiles) {
                GK_ASGB(1, true);  // d <= 128 on the tensor-core path
            } else if (d4 <= 32) {
                GK_ASGB(1, false);
            } else if (d4 <= 64) {
                GK_ASGB(2, false);
            } else if (d4 <= 128) {
                GK_ASGB(4, false);
            } else {
                GK_ASGB(8, false);
            }
#undef GK_ASGB
            done = true;
        }
    }
    if (done) {
    } else if (vec4 && d4 <= 32 * 8) {
#define GK_ASGG(NV, GS, LPR)                                                                                          \
    do {                                                                                                         \
        if (trk.dirty)                                                                                           \
            GK_ASGT(NV, GS, true, LPR);                                                                               \
        else                                                                                                     \
            GK_ASGT(NV, GS, false, LPR);                                                                              \
    } while (0)
#define GK_ASGT(NV, GS, T, LPR)                                                                                  \
    do {                                                                                                         \
        if ((e = resident_grid(reinterpret_cast<const void *>(k_assign_rows<NV, XT, GS, T, LPR>), AS_WARPS * 32, \
                               0, &grid)) != cudaSuccess)                                                        \
            return e;                                                                                            \
        k_assign_rows<NV, XT, GS, T, LPR><<<grid, AS_WARPS * 32, 0, s>>>(X, n, (int)d, ld, g_idx, kappa, C, k,   \
                                                                         labels_in, labels_out, best, st, trk,   \
                                                                         sel_lab);                               \
    } while (0)
#define GK_ASG(NV)                                                                                               \
    do {                                                                                                         \
        if constexpr (NV >= 8)                                                                                   \
            GK_ASGG(NV, 4, 32);                                                                                  \
        else if (gw == 4)                                                                                        \
            GK_ASGG(NV, 4, 32);                                                                                  \
        else                                                                                                     \
            GK_ASGG(NV, 8, 32);                                                                                  \
    } while (0)
        if (d4 <= 8)
            GK_ASGG(1, 4, 8);
        else if (d4 <= 16)
            GK_ASGG(1, 4, 16);
        else if (d4 <= 32)
            GK_ASG(1);
        else if (d4 <= 64)
            GK_ASG(2);
        else if (d4 <= 128)
            GK_ASG(4);
        else
            GK_ASG(8);
#undef GK_ASG
#undef GK_ASGG
#undef GK_ASGT
    } else {
        int dpad = (int)((d + 3) & ~3);
        size_t shm = sizeof(float) * (size_t)AS_WARPS * dpad + sizeof(int) * AS_WARPS * AS_QCAP;
        const int shm_max = (int)(sizeof(float) * (size_t)AS_WARPS * MAX_D + sizeof(int) * AS_WARPS * AS_QCAP);
        auto launch = [&](auto kernel) -> cudaError_t {
            cudaError_t le = set_max_smem(reinterpret_cast<const void *>(kernel), shm_max);
            if (le == cudaSuccess)
                kernel<<<AS_BLOCKS, AS_WARPS * 32, shm, s>>>(X, n, (int)d, ld, g_idx, kappa, C, k, labels_in, labels_out,
                                                             best, st, trk, sel_lab);
            return le;
        };
        if (vec4)
            e = trk.dirty ? launch(k_assign<4, XT, true>) : launch(k_assign<4, XT, false>);
        else
            e = trk.dirty ? launch(k_assign<1, XT, true>) : launch(k_assign<1, XT, false>);
        if (e != cudaSuccess)
            return e;
    }
    if (sum_d2 || n_changed || trk.dirty_out) {
        k_assign_reduce<<<AS_BLOCKS, 256, 0, s>>>(best, labels_in, labels_out, n, blk_sum, blk_chg, trk, k, sum_d2,
                                                  n_changed);
    }
    return cudaGetLastError();
}

cudaError_t launch_assign(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx,
                          int32_t kappa, const float *C, int32_t k, const int32_t *labels_in, int32_t *labels_out,
                          float *best_d2, double *sum_d2, int64_t *n_changed, void *scratch, DevStatus *st,
                          cudaStream_t s, int precision, const int32_t *members, Track trk)
{
    if (bf16)
        return assign_t(static_cast<const __nv_bfloat16 *>(X), n, d, ld, g_idx, kappa, C, k, labels_in, labels_out,
                        best_d2, sum_d2, n_changed, scratch, st, s, precision, members, trk);
    return assign_t(static_cast<const float *>(X), n, d, ld, g_idx, kappa, C, k, labels_in, labels_out, best_d2,
                    sum_d2, n_changed, scratch, st, s, precision, members, trk);
}

}  // namespace gkm
