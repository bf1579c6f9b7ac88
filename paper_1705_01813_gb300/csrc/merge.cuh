// Top-kappa merge of one graph row with a tile of candidates (Alg. 3: a
// compared pair updates the row), shared by the SIMT and tensor-core
// refinement kernels.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace gkm {

// A (distance, id) key packed in 64 bits so that one unsigned comparison
// orders keys as key_less does: the distance's bits mapped to an unsigned
// integer of the same order (sign bit set for non-negative values, all bits
// inverted for negative ones; -0 is first made +0, which compares equal to
// it) in the high word, the id (non-negative) in the low word.
__device__ __forceinline__ uint64_t pack_key(float dv, int id)
{
    const unsigned b = __float_as_uint(dv + 0.0f);
    const unsigned o = b ^ ((unsigned)((int)b >> 31) | 0x80000000u);
    return ((uint64_t)o << 32) | (uint32_t)id;
}

__device__ __forceinline__ float key_dist(uint64_t key)
{
    const unsigned o = (unsigned)(key >> 32);
    return __uint_as_float((o & 0x80000000u) ? (o ^ 0x80000000u) : ~o);
}

__device__ __forceinline__ int key_id(uint64_t key) { return (int)(uint32_t)key; }

// A graph row's kappa keys held in registers (lane l owns entries l, l + 32, ..., NU slots: 32 NU >= kappa), so that the
// next row's list can be loaded while the current row is merged.
template <int NU>
struct RowRegs {
    int id[NU];
    float dv[NU];
    int thi;  // the kappa-th key, in every lane
    float thd;
};

template <int NU>
__device__ __forceinline__ void load_row(RowRegs<NU> &r, const int32_t *__restrict__ gi, const float *__restrict__ gd,
                                         int kappa)
{
    const int lane = lane_id();
#pragma unroll
    for (int u = 0; u < NU; u++) {
        const int q = lane + 32 * u;
        if (q < kappa) {
            r.id[u] = __ldcg(gi + q);
            r.dv[u] = __ldcg(gd + q);
        }
    }
    r.thi = __ldcg(gi + kappa - 1);
    r.thd = __ldcg(gd + kappa - 1);
}

// The kernels that merge are compiled for each number of row slots: f(std::integral_constant<int, NU>) for this kappa.
template <typename F>
auto with_row_slots(int32_t kappa, F f)
{
    return kappa <= 32   ? f(std::integral_constant<int, 1>{})
           : kappa <= 64 ? f(std::integral_constant<int, 2>{})
                         : f(std::integral_constant<int, MAX_KAPPA / 32>{});
}

// Merging candidates into a graph row, warp-cooperative.  Lane l holds candidates l, l + 32, ... (NC slots) as packed
// keys ck[] with their flags ok[]: a candidate that beats the row's kappa-th key and is not the row itself, whose id
// may already be in the row.  The row's keys l, l + 32, ... (NU slots) come in `cur`.  Two forms with the same result:
//
// merge_few, for up to MERGE_FEW flagged candidates: one by one in registers.  A vote finds an id that is in the row
// (dropped); otherwise the row entries above the candidate move down one place, and the candidate's place is the row
// entries below it (ballots) plus the smaller candidates.  About 25 warp instructions a candidate, in a dependent
// chain of about 150 cycles, so only for a few.
//
// merge_many: the candidates are compacted, placed in the row by a binary search of a fixed number of steps, and
// ranked among themselves by comparing with all of them; their final places are marked in a bit mask, and every other
// place of the row takes the row entry that the mask counts off.  A candidate whose id is in the row is dropped: with
// `canon`, when the row's distances have the bits that the library computes for a pair (a graph that it built), its
// key is found at its place; otherwise the row ids are looked up among the candidates' ids (ascending, in shared
// memory).
//
// Only the entries that move are written; the result says whether a candidate entered the row.  Instruction issue bounds
// the merge: ranking, then binary searches for every candidate and row entry, took 1,400 warp instructions a row with 50
// candidates and 830 with 15; with these forms the merge of a 1M x 128 graph construction (kappa = 50) takes 0.64 ms a
// round instead of 0.94, the pairs left out included.
constexpr int MERGE_FEW = 4;

// Shared memory of one warp: the row's keys, the candidates' keys, repeat flags.
template <int NC>
struct alignas(16) MergeBuf {
    uint64_t rk[128], bk[32 * NC];
    unsigned dup[NC];
};

template <int NU, int NC>
__device__ __forceinline__ bool merge_few(uint64_t (&ck)[NC], bool (&ok)[NC], int kappa, const RowRegs<NU> &cur,
                                          int32_t *__restrict__ gi, float *__restrict__ gd)
{
    const int lane = lane_id();
    uint64_t rk[NU];
    int rid[NU], sh[NU];
#pragma unroll
    for (int u = 0; u < NU; u++) {
        const bool in = lane + 32 * u < kappa;
        rid[u] = in ? cur.id[u] : -1;
        rk[u] = in ? pack_key(cur.dv[u], cur.id[u]) : ~0ull;
        sh[u] = 0;
    }
    int rank[NC], pos[NC];
#pragma unroll
    for (int v = 0; v < NC; v++)
        rank[v] = pos[v] = 0;
#pragma unroll
    for (int v = 0; v < NC; v++) {
        unsigned bal = __ballot_sync(FULL_MASK, ok[v]);
        while (bal) {
            const int src = __ffs(bal) - 1;
            bal &= bal - 1;
            const uint64_t kb = __shfl_sync(FULL_MASK, ck[v], src);
            const int jb = key_id(kb);
            bool hit = false;
#pragma unroll
            for (int u = 0; u < NU; u++)
                hit |= rid[u] == jb;
            if (__any_sync(FULL_MASK, hit)) {
                if (lane == src)
                    ok[v] = false;
                continue;
            }
            int p = 0;
#pragma unroll
            for (int u = 0; u < NU; u++) {
                const bool lt = rk[u] < kb;
                p += __popc(__ballot_sync(FULL_MASK, lt));
                sh[u] += lt ? 0 : 1;
            }
#pragma unroll
            for (int c = 0; c < NC; c++)
                rank[c] += kb < ck[c] ? 1 : 0;
            if (lane == src)
                pos[v] = p;
        }
    }
#pragma unroll
    for (int u = 0; u < NU; u++) {
        const int q = lane + 32 * u + sh[u];
        if (sh[u] > 0 && q < kappa) {
            gi[q] = rid[u];
            gd[q] = key_dist(rk[u]);
        }
    }
    bool entered = false;
#pragma unroll
    for (int v = 0; v < NC; v++) {
        const int q = pos[v] + rank[v];
        if (ok[v] && q < kappa) {
            gi[q] = key_id(ck[v]);
            gd[q] = key_dist(ck[v]);
            entered = true;
        }
    }
    return __any_sync(FULL_MASK, entered);
}

// Number of the 32 N sorted keys k[] smaller than key (fixed steps; N a power of two).
template <int N>
__device__ __forceinline__ int lower_rank(const uint64_t *k, uint64_t key)
{
    int p = 0;
#pragma unroll
    for (int h = 16 * N; h >= 1; h >>= 1)
        p += k[p + h - 1] < key ? h : 0;
    return p + (k[p] < key ? 1 : 0);
}

// sid[0 .. ns): the ids of all candidate columns, ascending; smap[t] (NULL: t) the column of sid[t] (not read with
// canon).
template <int NU, int NC>
__device__ __forceinline__ bool merge_many(uint64_t (&ck)[NC], bool (&ok)[NC], bool canon, const int *__restrict__ sid,
                                           const unsigned char *__restrict__ smap, int ns, int kappa,
                                           const RowRegs<NU> &cur, int32_t *__restrict__ gi, float *__restrict__ gd,
                                           MergeBuf<NC> &mb)
{
    const int lane = lane_id();
    if (!canon) {
        if (lane < NC)
            mb.dup[lane] = 0u;
        __syncwarp();
    }
#pragma unroll
    for (int u = 0; u < NU; u++) {
        const int q = lane + 32 * u;
        uint64_t rk = ~0ull;
        if (q < kappa) {
            const int j = cur.id[u];
            rk = pack_key(cur.dv[u], j);
            if (!canon) {
                int p = 0;  // candidates with a smaller id
#pragma unroll
                for (int h = 16 * NC; h >= 1; h >>= 1)
                    p += p + h <= ns && sid[p + h - 1] < j ? h : 0;
                p += p < ns && sid[p] < j ? 1 : 0;
                if (p < ns && sid[p] == j) {
                    const int c = smap ? smap[p] : p;
                    atomicOr(&mb.dup[c >> 5], 1u << (c & 31));
                }
            }
        }
        mb.rk[q] = rk;
    }
    __syncwarp();
    int m = 0;
#pragma unroll
    for (int v = 0; v < NC; v++) {
        const bool o = ok[v] && (canon || ((mb.dup[v] >> lane) & 1u) == 0u);
        const unsigned bal = __ballot_sync(FULL_MASK, o);
        if (o)
            mb.bk[m + __popc(bal & lanemask_lt())] = ck[v];
        m += __popc(bal);
    }
    if (m == 0) {  // every candidate is in the row
        __syncwarp();
        return false;
    }
    if ((m & 1) && lane == 0)
        mb.bk[m] = ~0ull;  // the ranking loop reads pairs
    __syncwarp();
    uint64_t kb[NC];
    int f[NC];
#pragma unroll
    for (int v = 0; v < NC; v++) {
        f[v] = 0;
        kb[v] = ~0ull;
        if (32 * v < m) {
            const int b = lane + 32 * v;
            if (b < m) {
                kb[v] = mb.bk[b];
                f[v] = lower_rank<NU>(mb.rk, kb[v]);
                if (canon && mb.rk[f[v]] == kb[v])  // f < kappa: kb beats the row's last key
                    mb.bk[b] = kb[v] = ~0ull;       // already in the row: counts for nobody
            }
        }
    }
    __syncwarp();
    const ulonglong2 *b2 = reinterpret_cast<const ulonglong2 *>(mb.bk);
    if (NC == 1 || m <= 32) {
#pragma unroll 4
        for (int q = 0; q < (m + 1) / 2; q++) {
            const ulonglong2 w = b2[q];
            f[0] += (w.x < kb[0] ? 1 : 0) + (w.y < kb[0] ? 1 : 0);
        }
    } else {
#pragma unroll 2
        for (int q = 0; q < (m + 1) / 2; q++) {
            const ulonglong2 w = b2[q];
#pragma unroll
            for (int v = 0; v < NC; v++)
                f[v] += (w.x < kb[v] ? 1 : 0) + (w.y < kb[v] ? 1 : 0);
        }
    }
    unsigned mine[NU];
#pragma unroll
    for (int u = 0; u < NU; u++)
        mine[u] = 0u;
#pragma unroll
    for (int v = 0; v < NC; v++) {
        if (32 * v < m && kb[v] != ~0ull && f[v] < kappa) {
            gi[f[v]] = key_id(kb[v]);
            gd[f[v]] = key_dist(kb[v]);
#pragma unroll
            for (int u = 0; u < NU; u++)
                mine[u] |= (f[v] >> 5) == u ? 1u << (f[v] & 31) : 0u;
        }
    }
    int below = 0;
#pragma unroll
    for (int u = 0; u < NU; u++) {
        const unsigned mask = __reduce_or_sync(FULL_MASK, mine[u]);
        const int q = lane + 32 * u, a = q - below - __popc(mask & lanemask_lt());
        below += __popc(mask);
        if (q < kappa && a != q && ((mask >> lane) & 1u) == 0u) {
            const uint64_t key = mb.rk[a];
            gi[q] = key_id(key);
            gd[q] = key_dist(key);
        }
    }
    __syncwarp();  // the buffers are rewritten by the next row
    return below > 0;
}

// The form that the number of flagged candidates asks for.
template <int NU, int NC>
__device__ __forceinline__ bool merge_keys(uint64_t (&ck)[NC], bool (&ok)[NC], bool canon, const int *__restrict__ sid,
                                           const unsigned char *__restrict__ smap, int ns, int kappa,
                                           const RowRegs<NU> &cur, int32_t *__restrict__ gi, float *__restrict__ gd,
                                           MergeBuf<NC> &mb)
{
    int m = 0;
#pragma unroll
    for (int v = 0; v < NC; v++)
        m += __popc(__ballot_sync(FULL_MASK, ok[v]));
    if (m == 0)
        return false;
    if (m <= MERGE_FEW)
        return merge_few<NU, NC>(ck, ok, kappa, cur, gi, gd);
    return merge_many<NU, NC>(ck, ok, canon, sid, smap, ns, kappa, cur, gi, gd, mb);
}

// Merge a run's pair distances drow[0 .. ncol) (ncol <= 32 NC) to the members cid[] into graph row i of that run.
// crun[c] is the run that member c belonged to in the previous refinement (-1: none), irun the row's own: a pair
// that shared a run then has been offered to this row already, when it entered the row or lost to its kappa-th key,
// which has only decreased since, so it is left out here (its distance need not have been computed).  canon, sid, smap: see
// merge_many (the members in ascending id and the columns they have).
template <int NU, int NC>
__device__ __forceinline__ bool merge_row(int i, int irun, bool canon, const int *__restrict__ cid,
                                          const int *__restrict__ crun,
                                          const int *__restrict__ sid, const unsigned char *__restrict__ smap,
                                          const float *__restrict__ drow, int ncol, int kappa, const RowRegs<NU> &cur,
                                          int32_t *__restrict__ gi, float *__restrict__ gd, MergeBuf<NC> &mb)
{
    const int lane = lane_id();
    const uint64_t th = pack_key(cur.thd, cur.thi);
    uint64_t ck[NC];
    bool ok[NC];
#pragma unroll
    for (int v = 0; v < NC; v++) {
        const int c = lane + 32 * v;
        ck[v] = ~0ull;
        ok[v] = false;
        if (c < ncol) {
            const int j = cid[c];
            if (j >= 0 && j != i && (irun < 0 || crun[c] != irun)) {
                ck[v] = pack_key(drow[c], j);
                ok[v] = ck[v] < th;
            }
        }
    }
    return merge_keys<NU, NC>(ck, ok, canon, sid, smap, ncol, kappa, cur, gi, gd, mb);
}

}  // namespace gkm
