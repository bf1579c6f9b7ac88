// Graph refinement inside clusters (Alg. 3: every pair of samples that share
// a cluster is compared, and the pair's distance updates both samples' rows),
// exact FP32.
//
// A cluster of m members (CSR, ascending id) larger than max_cluster is cut
// into ceil(m / max_cluster) runs of consecutive members whose sizes differ by
// at most one; pairs are formed inside a run only.  k_refine_plan lists the
// runs; within a graph construction it leaves out those whose members all were
// in one run in the previous round, and the kernels below compare only pairs
// that were not: such a pair has been offered to both rows, and a kappa-th key
// only decreases, so it can neither be missing nor enter again (after the first
// round 1-67% of the pairs are new on the workloads' data; the refinements of a
// graph construction at 2M x 512 BF16 go from 62.1 to 16.4 ms, at 200k x 960
// FP32 from 16.3 to 12.9, at 1.3M x 64 in 16 jobs from 20.0 to 13.0).  A block
// takes a run: in a 64-wide tile where it has at most 64 members (the common
// case, several blocks per SM), in 128-wide tiles where it is longer.
// A run is covered by T x T tiles (rows x columns of the run); for each tile
// the block stages 32 coordinates of the row and column samples at a time in
// shared memory (the row samples twice over, as broadcast pairs) and every
// thread accumulates the pair distances of Q = T/16 consecutive rows and Q
// consecutive columns, two columns at a time in packed FP32x2 FMAs (the
// difference as fma(y, -1, x), then fma(e, e, acc): per pair the operations of
// pair_d2_seq), with one accumulator in ascending coordinate order, so a
// pair's distance has the same bits here, in the initial graph and in any
// later round.  Each warp then merges the tile's distances into the graph rows of its rows (merge.cuh).  Every
// row belongs to exactly one run per refinement, so blocks never write the
// same row.
#include "common.cuh"
#include "merge.cuh"
#include "tiles.cuh"

#include <type_traits>

namespace gkm {

// The runs of a refinement: int2 records {first position in the grouping, members}.  One array holds the runs of at
// most `split` members from its front (RunCounts::a of them) and the longer ones from its back (RunCounts::b).  A run
// whose members all shared one run in the previous refinement has no pair left to compare and is not listed.
constexpr int PL_WARPS = 8;

// One warp per `chunk` clusters (at most 32); the runs of a cluster that is cut are shared out over the block's warps
// (the SIFT- and GIST-shaped graphs grow clusters of thousands, 40 and 65 us a round with one warp each).  prev_in
// (may be NULL) and prev_out (may be NULL): per sample the run it
// belonged to in the previous and in this refinement, named by the run's first position; -1 for none.  The order in
// which runs are listed varies from call to call and decides nothing but which block takes a run.  This one kernel
// replaces counting the runs, scanning the counts and mapping runs to clusters (five launches, about 12 us a round).
__global__ void __launch_bounds__(PL_WARPS * 32) k_refine_plan(const int32_t *__restrict__ off,
                                                               const int32_t *__restrict__ mem, int64_t n, int k,
                                                               int cap, int split, int chunk,
                                                               const int32_t *__restrict__ prev_in,
                                                               int32_t *__restrict__ prev_out, int2 *__restrict__ runs,
                                                               int64_t runs_cap, RunCounts *__restrict__ cnt)
{
    __shared__ int s_ncut;
    __shared__ int2 s_cut[PL_WARPS * 32];  // {first member position, members} of the block's cut clusters
    const int lane = lane_id(), w = threadIdx.x >> 5;
    if (threadIdx.x == 0)
        s_ncut = 0;
    __syncthreads();
    const int64_t c0 = ((int64_t)blockIdx.x * PL_WARPS + w) * chunk;
    const int nq = (int)max((int64_t)0, min((int64_t)chunk, k - c0));
    int my_beg = 0, my_m = 0;
    if (lane < nq) {
        my_beg = off[c0 + lane];
        my_m = off[c0 + lane + 1] - my_beg;
        if (my_m > cap) {
            s_cut[atomicAdd(&s_ncut, 1)] = make_int2(my_beg, my_m);
            my_m = 0;
        }
    }
    // records the run of the members first .. first + sz - 1 in prev_out; has it a pair that was not compared before?
    auto visit = [&](int first, int sz) -> bool {
        bool same = prev_in != nullptr;
        if (same || prev_out) {
            int ref = -1;
#pragma unroll 2
            for (int t0 = 0; t0 < sz; t0 += 32) {
                const int t = t0 + lane;
                const int a = t < sz ? mem[first + t] : -1;
                const bool in = (unsigned)a < (unsigned)n;
                const int p = prev_in && in ? prev_in[a] : -1;
                if (t0 == 0)
                    ref = __shfl_sync(FULL_MASK, p, 0);
                same = same && (t >= sz || (p == ref && p >= 0));
                if (prev_out && in)
                    prev_out[a] = sz >= 2 ? first : -1;
            }
            same = __all_sync(FULL_MASK, same);
        }
        return sz >= 2 && !same;
    };
    int2 rec = make_int2(0, 0);
    // the lanes' records into the two lists, one atomic per list
    auto append = [&]() {
        const unsigned la = __ballot_sync(FULL_MASK, rec.y > 0 && rec.y <= split);
        const unsigned lb = __ballot_sync(FULL_MASK, rec.y > split);
        int ba = 0, bb = 0;
        if (lane == 0) {
            if (la)
                ba = atomicAdd(&cnt->a, __popc(la));
            if (lb)
                bb = atomicAdd(&cnt->b, __popc(lb));
        }
        ba = __shfl_sync(FULL_MASK, ba, 0);
        bb = __shfl_sync(FULL_MASK, bb, 0);
        if (rec.y > split)
            runs[runs_cap - 1 - (bb + __popc(lb & lanemask_lt()))] = rec;
        else if (rec.y > 0)
            runs[ba + __popc(la & lanemask_lt())] = rec;
        rec = make_int2(0, 0);
    };
    for (int q = 0; q < nq; q++) {
        const int beg = __shfl_sync(FULL_MASK, my_beg, q), m = __shfl_sync(FULL_MASK, my_m, q);
        if (m > 0 && visit(beg, m) && lane == q)
            rec = make_int2(beg, m);
    }
    append();
    __syncthreads();
    const int ncut = s_ncut;
    for (int z = 0; z < ncut; z++) {
        const int beg = s_cut[z].x, m = s_cut[z].y;
        const int nc = (m + cap - 1) / cap, base = m / nc, rem = m % nc;
        for (int b0 = 0; b0 < nc; b0 += PL_WARPS * 32) {
            for (int q = 0; q < 32; q++) {
                const int c = b0 + q * PL_WARPS + w;
                if (c >= nc)
                    break;
                const int first = beg + c * base + min(c, rem), sz = base + (c < rem ? 1 : 0);
                if (visit(first, sz) && lane == q)
                    rec = make_int2(first, sz);
            }
            append();
        }
    }
}

// Dynamic shared memory of k_refine: the stage buffers (the distance tile aliases them), ids and previous runs of the
// rows and columns, the members before they are sorted (a second id and run array), the list of blocks to compute.
template <int T>
__host__ __device__ constexpr size_t refine_smem_bytes()
{
    using TL = RefineTile<T>;
    return sizeof(float) * (TL::stage_floats > TL::tile_floats ? TL::stage_floats : TL::tile_floats) +
           sizeof(int) * 6 * T + T + sizeof(unsigned short) * ((TL::NBLK + 3) & ~3) + sizeof(int) * RF_WARPS +
           sizeof(MergeBuf<T / 32>) * RF_WARPS;
}

// The members of a run of sz <= T samples, read by the threads t < T of a group: ids (-1 for a corrupt entry, which is
// recorded, and past the end) and previous runs, in member order or, with prev, sorted by (previous run, member
// order), so that members that were together before are neighbours.  sid gets the ids in member order (ascending) and
// smap each one's place in rid (with prev only; else rid is in that order); spr: T entries of scratch.
template <int T, typename Sync>
__device__ __forceinline__ void load_members(const int32_t *__restrict__ S, int sz, int64_t n,
                                             const int32_t *__restrict__ prev, int *rid, int *rpr, int *sid,
                                             unsigned char *smap, int *spr, int t, int first, DevStatus *st, Sync sync)
{
    int a = -1, p = -1;
    if (t < T) {
        a = t < sz ? S[t] : -1;
        if (a >= n) {  // corrupt grouping: record, skip the sample
            flag_error(st, GK_ERR_INVALID, (unsigned)first);
            a = -1;
        }
        if (prev && a >= 0)
            p = prev[a];
        sid[t] = a;
        if (!prev || t >= sz) {
            rid[t] = a;
            rpr[t] = -1;
        }
    }
    if (prev) {
        if (t < T)
            spr[t] = p;
        sync();
        if (t < sz) {
            int r = 0;
            for (int q = 0; q < sz; q++)
                r += (spr[q] < p || (spr[q] == p && q < t)) ? 1 : 0;
            rid[r] = a;
            rpr[r] = p;
            smap[t] = (unsigned char)r;
        }
    }
    sync();
}

// Listed run blockIdx.x (longs: of the list from the back of the array) in T-wide tiles; the 64-wide instance gets runs of
// one tile only.  Registers bound it (the tile's accumulators, two rows' keys): compiled for the number of row slots
// NU, with the merge in one place and a run per block, it spills 28 bytes a thread (T = 64), 144 (T = 128) or none (T =
// 128, 16-byte loads).  With a choice of three NU inside and the merge inlined for runs of one tile and of several it
// spilled 208, 416 and 188: a refinement call of 1M x 960, k = 10,000 11.05 ms, now 9.36; 500k x 768 BF16, k = 5,000 4.56
// and 3.92; 1M x 128 at level 0 2.18 and 1.65 (kappa = 40; repeated calls 9.83 and 8.16, 3.94 and 3.30, 1.69 and 1.23).
template <int T, int NU, typename XT, bool VEC>
__global__ void __launch_bounds__(RF_THREADS, T == 64 ? 3 : 2) k_refine(const XT *__restrict__ X, int64_t n, int d,
                                                                        int64_t ld, const int32_t *__restrict__ mem,
                                                                        const int2 *__restrict__ runs,
                                                                        int64_t runs_cap,
                                                                        const RunCounts *__restrict__ cnt, bool longs,
                                                                        const int32_t *__restrict__ prev, bool canon,
                                                                        uint8_t *__restrict__ row_changed, int kappa,
                                                                        int32_t *__restrict__ g_idx,
                                                                        float *__restrict__ g_dist, DevStatus *st)
{
    using TL = RefineTile<T>;
    constexpr int DS = TL::DS, NC = T / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *xr = reinterpret_cast<float *>(smem_raw);  // staging buffers of the pair tiles (tiles.cuh)
    float *dt = xr;  // aliases the staging buffers
    constexpr size_t span = TL::stage_floats > TL::tile_floats ? TL::stage_floats : TL::tile_floats;
    int *rid = reinterpret_cast<int *>(xr + span);
    int *cid = rid + T, *rpr = cid + T, *cpr = rpr + T, *sid = cpr + T, *spr = sid + T;
    int *wcnt = spr + T;
    const int tid = threadIdx.x, w = tid >> 5;
    MergeBuf<NC> &mb = reinterpret_cast<MergeBuf<NC> *>(wcnt + RF_WARPS)[w];
    unsigned char *smap = reinterpret_cast<unsigned char *>(reinterpret_cast<MergeBuf<NC> *>(wcnt + RF_WARPS) + RF_WARPS);
    unsigned short *list = reinterpret_cast<unsigned short *>(smap + T);
    auto sync = [] { __syncthreads(); };
    if ((int)blockIdx.x >= (longs ? cnt->b : cnt->a))
        return;
    const int2 rec = longs ? runs[runs_cap - 1 - blockIdx.x] : runs[blockIdx.x];
    const int first = rec.x, sz = rec.y;
    const int32_t *S = mem + first;
    const bool one = T == 64 || sz <= T;  // one tile, whose members are sorted by their previous runs
    for (int rb = 0; rb < sz; rb += T) {
        const int nr = min(T, sz - rb);
        for (int cb = 0; cb < sz; cb += T) {
            const int ncl = min(T, sz - cb);
            __syncthreads();  // the previous tile's merges are done
            if (one) {
                load_members<T>(S, sz, n, prev, rid, rpr, sid, smap, spr, tid, first, st, sync);
            } else {
                for (int q = tid; q < T; q += RF_THREADS) {
                    int a = q < nr ? S[rb + q] : -1;
                    int b = q < ncl ? S[cb + q] : -1;
                    if (a >= n || b >= n) {  // corrupt grouping: record, skip the sample
                        flag_error(st, GK_ERR_INVALID, (unsigned)first);
                        a = a >= n ? -1 : a;
                        b = b >= n ? -1 : b;
                    }
                    rid[q] = a;
                    cid[q] = b;
                    rpr[q] = prev && a >= 0 ? prev[a] : -1;
                    cpr[q] = prev && b >= 0 ? prev[b] : -1;
                }
                __syncthreads();
            }
            if (rb == cb) {
                // the arithmetic goes to the block's warps rot, rot + 1, ... (rot = blockIdx.x % 4): each warp of an SM
                // issues on scheduler (its index % 4), so blocks that share an SM spread their few busy warps over all
                // four schedulers instead of all starting at scheduler 0
                const int t = (tid - (int)(blockIdx.x & 3) * 32) & (RF_THREADS - 1);
                int nlive, code;
                if (prev && one) {
                    nlive = live_blocks<T, RF_THREADS>(sz, rpr, list, wcnt, tid, sync);
                    code = t < nlive ? list[t] : 0;
                } else {
                    const int nb = (nr + TL::Q - 1) / TL::Q;
                    nlive = nb * (nb + 1) / 2;
                    code = t < nlive ? triangle_block(nb, t) : 0;
                }
                tile_distances<T, true, VEC>(X, d, ld, rid, rid, code >> 8, code & 255, t < nlive, xr, dt);
            } else {
                tile_distances<T, false, VEC>(X, d, ld, rid, cid, tid >> 4, tid & 15, TL::Q * (tid >> 4) < nr, xr, dt);
            }
            __syncthreads();
            const int *ci = one ? rid : cid, *cp = one ? rpr : cpr, *si = one ? sid : cid;
            const unsigned char *sm = one && prev ? smap : nullptr;
            RowRegs<NU> cur, nxt;
            if (w < nr && rid[w] >= 0)
                load_row(cur, g_idx + (int64_t)rid[w] * kappa, g_dist + (int64_t)rid[w] * kappa, kappa);
            for (int row = w; row < nr; row += RF_WARPS) {
                const int i = rid[row];
                const int rn = row + RF_WARPS;
                if (rn < nr && rid[rn] >= 0)  // next row's list in flight during this merge
                    load_row(nxt, g_idx + (int64_t)rid[rn] * kappa, g_dist + (int64_t)rid[rn] * kappa, kappa);
                if (i >= 0 && merge_row<NU, NC>(i, rpr[row], canon, ci, cp, si, sm, dt + row * DS, ncl, kappa, cur,
                                                g_idx + (int64_t)i * kappa, g_dist + (int64_t)i * kappa, mb) &&
                    row_changed && lane_id() == 0)
                    row_changed[i] = 1;
                cur = nxt;
            }
        }
    }
}

// Listed runs of at most 64 members, warp-specialised: a persistent block takes runs blockIdx.x, + gridDim.x, ...; five
// of its nine warps (the compute group, WS_NC threads, rotated over the block's warps by blockIdx.x so that the
// blocks of an SM spread them over its four schedulers) stage and compute a run's pair tile while the other four
// merge the previous run's rows.  The two hand the distance tile over through named barriers: FULL (the compute group
// arrives when the tile and the run's ids are written, the merge warps wait) and EMPTY (the merge warps arrive
// when they no longer read it, the compute group waits before writing the next one).  Both sides walk the same
// list, so the barriers pair up: per run one FULL and one EMPTY phase, plus the EMPTY phase
// the merge warps open before the first run and the compute group closes after the last.  Pair arithmetic,
// merge order and results are those of k_refine<64>.
constexpr int WS_NC = 160;  // compute group: 5 warps, covers the 136 pair blocks of a 64-row triangle
constexpr int WS_NM = 4;    // merge warps
constexpr int WS_THREADS = WS_NC + 32 * WS_NM;
constexpr int WS_BAR_C = 1, WS_BAR_FULL = 2, WS_BAR_EMPTY = 3;

// dynamic shared memory: two stage buffers, the distance tile, two runs' members (ids and previous runs, ids in
// member order and their places), scratch of the sort, the merge warps' buffers, the list of blocks to compute
__host__ __device__ constexpr size_t refine_ws_smem_bytes()
{
    using TL = RefineTile<64>;
    return sizeof(float) * (TL::stage_floats + TL::tile_floats) + sizeof(int) * 7 * 64 + 2 * 64 +
           sizeof(int) * 8 + sizeof(MergeBuf<2>) * WS_NM + sizeof(unsigned short) * ((TL::NBLK + 3) & ~3);
}

template <int NU, typename XT, bool VEC>
__global__ void __launch_bounds__(WS_THREADS, 3) k_refine_ws(const XT *__restrict__ X, int64_t n, int d, int64_t ld,
                                                             const int32_t *__restrict__ mem,
                                                             const int2 *__restrict__ runs,
                                                             const RunCounts *__restrict__ cnt,
                                                             const int32_t *__restrict__ prev, bool canon,
                                                                        uint8_t *__restrict__ row_changed, int kappa,
                                                             int32_t *__restrict__ g_idx,
                                                             float *__restrict__ g_dist, DevStatus *st)
{
    constexpr int T = 64;
    using TL = RefineTile<T>;
    constexpr int DS = TL::DS, Q = TL::Q;
    constexpr int WARPS = WS_THREADS / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *stage = reinterpret_cast<float *>(smem_raw);
    float *dt = stage + TL::stage_floats;
    int *rids = reinterpret_cast<int *>(dt + TL::tile_floats);  // [2][T]: the ids of runs j and j + 1
    int *rprs = rids + 2 * T;                                   // [2][T]: their previous runs
    int *sids = rprs + 2 * T;                                   // [2][T]: the ids in member order
    int *spr = sids + 2 * T, *wcnt = spr + T;
    MergeBuf<2> *mbufs = reinterpret_cast<MergeBuf<2> *>(wcnt + 8);
    unsigned char *smaps = reinterpret_cast<unsigned char *>(mbufs + WS_NM);  // [2][T]: and their places
    unsigned short *list = reinterpret_cast<unsigned short *>(smaps + 2 * T);
    const int w = threadIdx.x >> 5, lane = lane_id();
    const int rr = (w + WARPS - (int)(blockIdx.x & 3)) % WARPS;  // 0 .. 4: compute group, 5 .. 8: merge warps
    const int nrun = cnt->a;
    if (rr < 5) {
        // ---- compute group ----
        const int ct = rr * 32 + lane;
        auto sync = [] { bar_sync(WS_BAR_C, WS_NC); };
        int j = 0;
        for (int run = blockIdx.x; run < nrun; run += gridDim.x) {
            const int2 rec = runs[run];
            // the merges of run j - 2, which read this slot, ended before EMPTY of run j - 1
            int *rid = rids + (j & 1) * T, *rpr = rprs + (j & 1) * T;
            load_members<T>(mem + rec.x, rec.y, n, prev, rid, rpr, sids + (j & 1) * T, smaps + (j & 1) * T, spr, ct, rec.x,
                            st, sync);
            int nlive, code;
            if (prev) {
                nlive = live_blocks<T, WS_NC>(rec.y, rpr, list, wcnt, ct, sync);
                code = ct < nlive ? list[ct] : 0;
            } else {
                const int nb = (rec.y + Q - 1) / Q;
                nlive = nb * (nb + 1) / 2;
                code = ct < nlive ? triangle_block(nb, ct) : 0;
            }
            const bool live = ct < nlive;
            const int by = code >> 8, bx = code & 255;
            float2 acc[Q][Q / 2];
            tile_distances_group<WS_NC, VEC>(X, d, ld, rid, by, bx, live, stage, ct, WS_BAR_C, acc);
            bar_sync(WS_BAR_EMPTY, WS_THREADS);  // the merge warps no longer read the distance tile
            if (live) {
#pragma unroll
                for (int a = 0; a < Q; a++)
#pragma unroll
                    for (int b = 0; b < Q / 2; b++) {
                        dt[(Q * by + a) * DS + Q * bx + 2 * b] = acc[a][b].x;
                        dt[(Q * by + a) * DS + Q * bx + 2 * b + 1] = acc[a][b].y;
                        if (by != bx) {
                            dt[(Q * bx + 2 * b) * DS + Q * by + a] = acc[a][b].x;
                            dt[(Q * bx + 2 * b + 1) * DS + Q * by + a] = acc[a][b].y;
                        }
                    }
            }
            __threadfence_block();
            bar_arrive(WS_BAR_FULL, WS_THREADS);  // this run's ids and distance tile are in place
            j++;
        }
        bar_sync(WS_BAR_EMPTY, WS_THREADS);  // the merge warps' arrival after the last run
    } else {
        // ---- merge warps ----
        const int mw = rr - 5;
        bar_arrive(WS_BAR_EMPTY, WS_THREADS);  // the distance tile starts free
        int j = 0;
        for (int run = blockIdx.x; run < nrun; run += gridDim.x) {
            const int sz = runs[run].y;
            const int *rid = rids + (j & 1) * T, *rpr = rprs + (j & 1) * T;
            const int *sid = sids + (j & 1) * T;
            const unsigned char *smap = prev ? smaps + (j & 1) * T : nullptr;
            bar_sync(WS_BAR_FULL, WS_THREADS);  // run j's ids and distances
            RowRegs<NU> cur, nxt;
            if (mw < sz && rid[mw] >= 0)
                load_row(cur, g_idx + (int64_t)rid[mw] * kappa, g_dist + (int64_t)rid[mw] * kappa, kappa);
            for (int row = mw; row < sz; row += WS_NM) {
                const int i = rid[row];
                const int rn = row + WS_NM;
                if (rn < sz && rid[rn] >= 0)  // next row's list in flight during this merge
                    load_row(nxt, g_idx + (int64_t)rid[rn] * kappa, g_dist + (int64_t)rid[rn] * kappa, kappa);
                if (i >= 0 && merge_row<NU, T / 32>(i, rpr[row], canon, rid, rpr, sid, smap, dt + row * DS, sz, kappa, cur,
                                                g_idx + (int64_t)i * kappa, g_dist + (int64_t)i * kappa, mbufs[mw]) &&
                    row_changed && lane == 0)
                    row_changed[i] = 1;
                cur = nxt;
            }
            __threadfence_block();
            bar_arrive(WS_BAR_EMPTY, WS_THREADS);  // done with the distance tile and this slot of ids
            j++;
        }
    }
}

// runs per refinement: sum over clusters of ceil(m / max_cluster), at most k + n / max_cluster (max_cluster >= 2)
static int64_t max_runs(int64_t n, int32_t k) { return (int64_t)k + n / 2 + 1; }
static size_t runs_bytes(int64_t n, int32_t k) { return ((size_t)max_runs(n, k) * sizeof(int2) + 255) / 256 * 256; }

size_t refine_scratch_bytes(int64_t n, int32_t k, int64_t d)
{
    return 256 + runs_bytes(n, k) + refine_tc_scratch_bytes(n, k, d);
}

template <typename XT, bool VEC>
static cudaError_t refine_tv(const XT *X, int64_t n, int64_t d, int64_t ld, const int32_t *offsets,
                             const int32_t *members, int32_t k, int32_t kappa, int32_t max_cluster, int32_t *g_idx,
                             float *g_dist, void *scratch, DevStatus *st, cudaStream_t s, int precision,
                             const int32_t *prev_in, int32_t *prev_out, bool canon, uint8_t *row_changed)
{
    RunCounts *cnt = static_cast<RunCounts *>(scratch);
    int2 *runs = reinterpret_cast<int2 *>(static_cast<char *>(scratch) + 256);
    void *tc_scratch = static_cast<char *>(scratch) + 256 + runs_bytes(n, k);
    const int64_t runs_cap = max_runs(n, k);
    cudaError_t e;
    // The tensor-core path for 64 <= d <= 128.  Its Gram is exact only for integer data with 2 d 255^2 < 2^24
    // (d <= 128), and wider rows made the recompute of every kept pair dearer than the FP32 tile kernels
    // (1M x 960 FP32: 91 ms against 25 ms per call; 10M x 512 BF16 unit vectors, whose Gram carries no BF16
    // rounding but of whose pairs about 45% may enter a row in every round: 106 ms against 86 ms); for d < 64 the
    // tile kernels'
    // cost, proportional to d, is below the fixed per-run cost of the Gram path (20k x 32: 0.18 ms against
    // 0.12 ms per call).
    const bool tensor = precision >= 1 && d >= 64 && d <= 128;
    const int split = tensor ? 128 : 64;
    if ((e = cudaMemsetAsync(cnt, 0, sizeof(RunCounts), s)) != cudaSuccess)
        return e;
    // clusters per warp: enough warps to fill the chip first, then fewer atomics on the list counters
    const int64_t per = k / (152 * 32);
    const int chunk = per < 1 ? 1 : per > 32 ? 32 : (int)per;
    const int64_t pblocks = ((int64_t)k + (int64_t)chunk * PL_WARPS - 1) / ((int64_t)chunk * PL_WARPS);
    k_refine_plan<<<(unsigned)pblocks, PL_WARPS * 32, 0, s>>>(offsets, members, n, k, max_cluster, split, chunk, prev_in,
                                                              prev_out, runs, runs_cap, cnt);
    // an upper bound of the number of runs: sum over clusters of (m / cap + 1)
    const int64_t bound = (int64_t)k + n / max_cluster + 1;
    auto blocks = [&](int resident) { return (unsigned)(bound < resident ? bound : resident); };
    // a block per run, handed out as blocks finish (a wave of blocks walking the list was 4% slower)
    // runs of more than `split` members (FP32 tiles of 128; longer runs in several tiles)
    if (max_cluster > split) {
        constexpr size_t shm = refine_smem_bytes<128>();
        auto kernel = with_row_slots(kappa, [](auto nu) { return k_refine<128, decltype(nu)::value, XT, VEC>; });
        const void *f = reinterpret_cast<const void *>(kernel);
        if ((e = set_max_smem(f, (int)shm)) != cudaSuccess)
            return e;
        kernel<<<(unsigned)bound, RF_THREADS, shm, s>>>(X, n, (int)d, ld, members, runs, runs_cap, cnt, true, prev_in,
                                                        canon, row_changed, kappa, g_idx, g_dist, st);
    }
    if (tensor) {
        // tensor-core Gram for runs of <= 128 members
        constexpr bool bf16 = std::is_same_v<XT, __nv_bfloat16>;
        return launch_refine_tc(X, bf16, n, d, ld, members, runs, cnt, bound, k, kappa, prev_in, canon, row_changed, g_idx,
                                g_dist, tc_scratch, st, s);
    }
    // runs of <= 64 members.  Rows staged by
    // 16-byte loads take the persistent warp-specialised kernel (one wave of blocks; 10M x 512 BF16: 32.0 ->
    // 31.3 ms per call, 98 -> 75 ms for runs of about ten); rows staged element by element keep the plain block,
    // where five warps' share of the element loads made the specialised form slower (1M x 960 FP32: 7.6
    // against 7.7 ms; 1M x 128 FP32: 3.7 against 3.9 ms)
    if constexpr (VEC) {
        int grid = 0;
        constexpr size_t shm = refine_ws_smem_bytes();
        auto kernel = with_row_slots(kappa, [](auto nu) { return k_refine_ws<decltype(nu)::value, XT, VEC>; });
        const void *f = reinterpret_cast<const void *>(kernel);
        if ((e = set_max_smem(f, (int)shm)) != cudaSuccess || (e = resident_grid(f, WS_THREADS, shm, &grid)) != cudaSuccess)
            return e;
        kernel<<<blocks(grid), WS_THREADS, shm, s>>>(X, n, (int)d, ld, members, runs, cnt, prev_in, canon, row_changed,
                                                     kappa, g_idx, g_dist, st);
    } else {
        constexpr size_t shm = refine_smem_bytes<64>();
        auto kernel = with_row_slots(kappa, [](auto nu) { return k_refine<64, decltype(nu)::value, XT, VEC>; });
        const void *f = reinterpret_cast<const void *>(kernel);
        if ((e = set_max_smem(f, (int)shm)) != cudaSuccess)
            return e;
        kernel<<<(unsigned)bound, RF_THREADS, shm, s>>>(X, n, (int)d, ld, members, runs, runs_cap, cnt, false, prev_in,
                                                        canon, row_changed, kappa, g_idx, g_dist, st);
    }
    return cudaGetLastError();
}

// the tile kernels with 16-byte stage loads where the rows allow them, for BF16 rows (eight elements per load
// instead of one 2-byte load each; FP32 rows keep the element loads, whose kernel uses fewer registers)
template <typename XT>
static cudaError_t refine_t(const XT *X, int64_t n, int64_t d, int64_t ld, const int32_t *offsets,
                            const int32_t *members, int32_t k, int32_t kappa, int32_t max_cluster, int32_t *g_idx,
                            float *g_dist, void *scratch, DevStatus *st, cudaStream_t s, int precision,
                            const int32_t *prev_in, int32_t *prev_out, bool canon, uint8_t *row_changed)
{
    if constexpr (std::is_same_v<XT, __nv_bfloat16>)
        if (tile_vec16(X, (int)d, ld))
            return refine_tv<XT, true>(X, n, d, ld, offsets, members, k, kappa, max_cluster, g_idx, g_dist, scratch, st,
                                       s, precision, prev_in, prev_out, canon, row_changed);
    return refine_tv<XT, false>(X, n, d, ld, offsets, members, k, kappa, max_cluster, g_idx, g_dist, scratch, st, s,
                                precision, prev_in, prev_out, canon, row_changed);
}

cudaError_t launch_refine(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *offsets,
                          const int32_t *members, int32_t k, int32_t kappa, int32_t max_cluster, int32_t *g_idx,
                          float *g_dist, void *scratch, DevStatus *st, cudaStream_t s, int precision,
                          const int32_t *prev_in, int32_t *prev_out, bool canon, uint8_t *row_changed)
{
    if (bf16)
        return refine_t(static_cast<const __nv_bfloat16 *>(X), n, d, ld, offsets, members, k, kappa, max_cluster,
                        g_idx, g_dist, scratch, st, s, precision, prev_in, prev_out, canon, row_changed);
    return refine_t(static_cast<const float *>(X), n, d, ld, offsets, members, k, kappa, max_cluster, g_idx, g_dist,
                    scratch, st, s, precision, prev_in, prev_out, canon, row_changed);
}

}  // namespace gkm
