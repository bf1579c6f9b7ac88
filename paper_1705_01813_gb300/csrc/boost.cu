// Boost form of GK-means (Sec. 3.1 Eq. 2 and Eq. 3; the move step of Alg. 2,
// Sec. 4.2).  State per cluster r: the composite vector D_r (FP64, the sum of
// its members, Eq. 2), its size n_r and S_r = D_r'D_r.  Alg. 2 visits samples
// one at a time; sample i in cluster u looks at the clusters of its kappa
// neighbours and moves to the one whose Eq. 3 gain
//     ((D_v + x)'(D_v + x) / (n_v + 1) + (D_u - x)'(D_u - x) / (n_u - 1)) - S_v / n_v - S_u / n_u
// is largest, if that gain is positive.  Each move changes two clusters and one
// label before the next visit reads them, so the result is that of visiting in
// order; the kernel below evaluates windows of visits at once and commits them
// in order only as far as that result allows.
//
// Arithmetic, fixed so that every decision is reproducible: FP64; D_r starts
// as its members' rows summed in ascending sample id; a squared norm squares
// the elements (each rounded once) of the vector zero-padded to a power of two
// and sums them by halving folds (w[j] += w[j + P/2], then P/4, ...); the gain
// is evaluated term by term, left to right, every operation rounded once (no
// fused multiply-add).  A sample alone in its cluster does not move (Eq. 3
// divides by n_u - 1); equal gains go to the smaller label.
//
// Layout: D is k x d row-major FP64; S, counts and labels are k / k / n
// arrays.  One thread-block cluster (up to 16 CTAs, one per SM) runs the
// epoch.  GB300 runs FP64 at a small fraction of its FP32 rate, so the tasks
// are screened in FP32 and few are folded in FP64.  After a move, S_u and S_v
// are the two norms computed for the decision: the new rows are exactly the
// rounded sums that were squared.
#include <climits>
#include <map>
#include <mutex>

#include "common.cuh"

namespace gkm {

namespace {

constexpr int BO_MAX_D = 1024;

// Squared norm of a lane-major vector (lane l holds w[l + 32 m], m < PL) by
// halving folds; the total lands in lane 0.  Folds with a stride of 32 or more
// stay inside a lane; the last five are shuffles.
template <int PL>
__device__ __forceinline__ double fold_lanes(double (&w)[PL])
{
#pragma unroll
    for (int h = PL / 2; h >= 1; h /= 2)
#pragma unroll
        for (int m = 0; m < h; m++)
            w[m] = __dadd_rn(w[m], w[m + h]);
    double a = w[0];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
        a = __dadd_rn(a, __shfl_down_sync(FULL_MASK, a, o));
    return a;
}

template <typename XT>
__device__ __forceinline__ double ldx64(const XT *p)
{
    return widen(ldx(p));
}

// ---------------------------------------------------------------------------
// Eq. 2 state from a CSR grouping (members ascending within a cluster).
// ---------------------------------------------------------------------------
constexpr int BS_THREADS = 128;

// D[r][t]: one thread per (cluster, coordinate), members summed in CSR order.
template <typename XT>
__global__ void __launch_bounds__(BS_THREADS) k_boost_sum(const XT *__restrict__ X, int d, int64_t ld,
                                                         const int32_t *__restrict__ offsets,
                                                         const int32_t *__restrict__ members, double *__restrict__ D)
{
    const int r = blockIdx.x;
    const int t = blockIdx.y * BS_THREADS + threadIdx.x;
    if (t >= d)
        return;
    const int b = offsets[r], e = offsets[r + 1];
    double acc = 0.0;
    int p = b;
    for (; p + 4 <= e; p += 4) {  // loads issued ahead of the ordered additions
        const double a0 = ldx64(X + (int64_t)members[p] * ld + t), a1 = ldx64(X + (int64_t)members[p + 1] * ld + t);
        const double a2 = ldx64(X + (int64_t)members[p + 2] * ld + t), a3 = ldx64(X + (int64_t)members[p + 3] * ld + t);
        acc = __dadd_rn(__dadd_rn(__dadd_rn(__dadd_rn(acc, a0), a1), a2), a3);
    }
    for (; p < e; p++)
        acc = __dadd_rn(acc, ldx64(X + (int64_t)members[p] * ld + t));
    D[(int64_t)r * d + t] = acc;
}

// S[r] = D_r'D_r (the fold) and counts[r], one warp per cluster.
template <int PL>
__global__ void __launch_bounds__(256) k_boost_norms(const double *__restrict__ D, int d, int32_t k,
                                                     const int32_t *__restrict__ offsets, double *__restrict__ S,
                                                     int32_t *__restrict__ counts)
{
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= k)
        return;
    const int lane = lane_id();
    double w[PL];
#pragma unroll
    for (int m = 0; m < PL; m++) {
        const int j = lane + 32 * m;
        const double a = j < d ? D[(int64_t)r * d + j] : 0.0;
        w[m] = __dmul_rn(a, a);
    }
    const double s = fold_lanes<PL>(w);
    if (lane == 0) {
        S[r] = s;
        counts[r] = offsets[r + 1] - offsets[r];
    }
}

// ---------------------------------------------------------------------------
// One epoch of the move step over order[0..m), on one cluster of R CTAs, in
// windows of up to W visits.
//
// A window's visits are evaluated together against the state at its start,
// visit j on CTA j mod R: the CTA gathers the visit's candidate set and screens
// every (visit, cluster) task in FP32, one warp per task.  With S_r = D_r'D_r
// the two halves of the gain are
//   (2 D_v'x + x'x - S_v / n_v) / (n_v + 1)   and   (x'x - 2 D_u'x + S_u / n_u) / (n_u - 1),
// so a dot product gives them to (PL + 16) 2^-23 of their terms' sizes, and an
// interval per candidate.  Only the candidates whose interval reaches the
// largest lower end, and only where the gain can be positive, are evaluated as
// defined (the FP64 folds and quotients); the arg-max over those is the arg-max
// over all.  Whatever leaves FP32's comfortable range, or is no number, has an
// unbounded interval and is evaluated as defined.
//
// Each CTA writes its visits' moves into every CTA of the cluster.  The window
// commits in order up to the first visit whose inputs an earlier moving visit
// changed (its sample or one of its neighbours moved; its own cluster or a
// candidate was the source or target of a move), which each CTA looks up for
// its own visits.  A committed visit therefore saw exactly the state the
// sequential walk gives it, and the committed moves touch disjoint clusters, so
// each CTA applies its own; the next window starts at the first visit not
// committed (the first visit of a window always commits).  The three cluster
// barriers of a window are unconditional.  Mutable state (labels, D, S, counts)
// is read through L2 (ld.global.cg), which the barriers order; samples and graph
// rows of the next window are on their way during the last barrier.
//
// Bound by the chain of a window's dependent steps (loads, barriers), so every
// window takes all W visits: 8.5 against 9.2 ms for 20,000 visits when the
// window shrinks after a cut, 10.6 with 16 visits.  At 1M x 128, k = 10,000,
// kappa = 50 (a quarter of the visits move) 0.43 us a visit; with every task
// folded in FP64 and gains and commit on one CTA it was 1.74 (the folds' FP64
// work 0.7, one CTA's part and everyone's loading of all visits the rest).
// 256 or 1024 threads, and 2 or 8 tasks of a warp at once: 2-4% slower.
// ---------------------------------------------------------------------------
constexpr int BE_THREADS = 512;
constexpr int BE_WARPS = BE_THREADS / 32;
constexpr int BE_MAX_CLUSTER = 16;
constexpr int BE_MAX_WINDOW = 32;  // a lane per visit
constexpr size_t BE_SMEM_BUDGET = 200 * 1024;

// An FP64 value cut to FP32 on the integer pipe (the FP64 one is narrow): error below 2^-23 of it, 0 below FP32's
// normal range, NaN above it.
__device__ __forceinline__ float cut32(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v), a = hi & 0x7fffffffu;
    const unsigned f = (hi & 0x80000000u) | ((__funnelshift_l(lo, hi, 3) & 0x7fffffffu) ^ 0x40000000u);
    return a < 0x38100000u ? 0.f : __uint_as_float(a < 0x47f00000u ? f : 0x7fc00000u);
}

// Dynamic shared memory of one CTA for windows of W visits (the same layout in every CTA of the cluster).  V: the
// CTA's visits; task c of its visit q is entry q (kp + 1) + c, c = 0 the own cluster.
struct WinLayout {
    int W, V, kp;
    size_t xs, sg, sq, tg, te, tm, ea, es, en, tl, svis, su, snq, sxx, nev, nat, mve, mvi, mvu, mvv, dep, bytes;
    __host__ __device__ WinLayout(int W_, int P, int kappa, int R)
    {
        W = W_;
        V = (W + R - 1) / R;
        kp = (kappa + 31) / 32 * 32;
        const int TM = V * (kp + 1);
        size_t o = 0;
        auto take = [&](size_t bytes) {
            const size_t at = o;
            o += (bytes + 15) / 16 * 16;
            return at;
        };
        xs = take((size_t)V * P * 4);
        sg = take((size_t)V * kp * 4);
        sq = take((size_t)V * kp * 4);
        tg = take((size_t)TM * 4);
        te = take((size_t)TM * 4);
        tm = take((size_t)TM * 4);
        ea = take((size_t)TM * 8);
        es = take((size_t)TM * 8);
        en = take((size_t)TM * 4);
        tl = take((size_t)TM * 4);
        svis = take((size_t)V * 4);
        su = take((size_t)V * 4);
        snq = take((size_t)V * 4);
        sxx = take((size_t)V * 4);
        nev = take((size_t)V * 4);
        nat = take((size_t)V * 4);
        mve = take((size_t)V * 4);
        mvi = take((size_t)W * 4);
        mvu = take((size_t)W * 4);
        mvv = take((size_t)W * 4);
        dep = take((size_t)W * 4);
        bytes = o;
    }
};

template <typename XT, int PL>
__global__ void __launch_bounds__(BE_THREADS, 1)
    k_boost_epoch(const XT *__restrict__ X, int32_t n, int d, int64_t ld, const int32_t *__restrict__ G, int kappa,
                  const int32_t *__restrict__ order, int64_t m, int32_t *L, int32_t k, double *D, int32_t *cnt,
                  double *S, int64_t *n_moved, DevStatus *st, int W)
{
    constexpr int P = 32 * PL;
    constexpr int B = PL <= 4 ? 4 : PL == 8 ? 2 : 1;  // screening tasks of a warp whose rows are in flight together
    constexpr int KC = MAX_KAPPA / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_ne;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int rank = (int)cluster_rank(), R = (int)cluster_size();
    const WinLayout Y(W, P, kappa, R);
    const int kp = Y.kp, ks = kp + 1;
    float *xs = reinterpret_cast<float *>(smem + Y.xs);
    int *sg = reinterpret_cast<int *>(smem + Y.sg), *sq = reinterpret_cast<int *>(smem + Y.sq);
    float *tg = reinterpret_cast<float *>(smem + Y.tg), *te = reinterpret_cast<float *>(smem + Y.te);
    float *tm = reinterpret_cast<float *>(smem + Y.tm);
    double *ea = reinterpret_cast<double *>(smem + Y.ea), *es = reinterpret_cast<double *>(smem + Y.es);
    int *en = reinterpret_cast<int *>(smem + Y.en), *tl = reinterpret_cast<int *>(smem + Y.tl);
    int *svis = reinterpret_cast<int *>(smem + Y.svis), *su = reinterpret_cast<int *>(smem + Y.su);
    int *snq = reinterpret_cast<int *>(smem + Y.snq), *nev = reinterpret_cast<int *>(smem + Y.nev);
    float *sxx = reinterpret_cast<float *>(smem + Y.sxx);
    int *nat = reinterpret_cast<int *>(smem + Y.nat), *mve = reinterpret_cast<int *>(smem + Y.mve);
    int *mvi = reinterpret_cast<int *>(smem + Y.mvi), *mvu = reinterpret_cast<int *>(smem + Y.mvu);
    int *mvv = reinterpret_cast<int *>(smem + Y.mvv), *dep = reinterpret_cast<int *>(smem + Y.dep);
    int64_t moves = 0;

    // the visits of a window from position s on, what no move changes: ids, samples, graph rows (one warp per visit)
    auto fetch = [&](int64_t s, int Wn) {
        for (int q = w; q * R + rank < Wn; q += BE_WARPS) {
            const int64_t at = s + q * R + rank;
            const int i = __ldg(order + at);
            const bool ok = i >= 0 && i < n;
            if (!ok && lane == 0)
                flag_error(st, GK_ERR_INVALID, (unsigned)at);
            int g[KC];
#pragma unroll
            for (int c = 0; c < KC; c++)
                g[c] = ok && 32 * c + lane < kappa ? __ldg(G + (int64_t)i * kappa + 32 * c + lane) : -1;
            float x[PL], xx = 0.f;
#pragma unroll
            for (int p = 0; p < PL; p++)
                x[p] = ok && lane + 32 * p < d ? ldx(X + (int64_t)i * ld + lane + 32 * p) : 0.f;
#pragma unroll
            for (int c = 0; c < KC; c++)
                if (32 * c < kp)
                    sg[q * kp + 32 * c + lane] = g[c];
#pragma unroll
            for (int p = 0; p < PL; p++) {
                xs[q * P + lane + 32 * p] = x[p];
                xx = fmaf(x[p], x[p], xx);
            }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1)
                xx += __shfl_xor_sync(FULL_MASK, xx, o);
            if (lane == 0) {
                svis[q] = ok ? i : -1;
                sxx[q] = xx;
            }
        }
        __syncwarp();
    };
    int Wn = (int)(m < (int64_t)W ? m : (int64_t)W);
    cluster_arrive();  // every CTA of the cluster runs before any stores into another's shared memory
    fetch(0, Wn);
    cluster_wait();

    for (int64_t s = 0; s < m;) {
        const int nv = Wn > rank ? (Wn - rank + R - 1) / R : 0;  // this CTA's visits
        if (threadIdx.x == 0)
            s_ne = 0;
        // ---- labels and candidate set of visit q, distinct labels other than its own, by the warp that fetched it
        for (int q = w; q < nv; q += BE_WARPS) {
            const int i = svis[q];  // written by this warp's lane 0 before a barrier
            int u = -1, lab[KC];
            if (i >= 0)
                u = __ldcg(L + i);
#pragma unroll
            for (int c = 0; c < KC; c++) {
                lab[c] = -3;  // no label wanted
                if (i >= 0 && 32 * c + lane < kappa) {
                    const int g = sg[q * kp + 32 * c + lane];
                    lab[c] = g >= 0 && g < n ? __ldcg(L + g) : -2;
                }
            }
            if (i >= 0 && (u < 0 || u >= k)) {
                if (lane == 0)
                    flag_error(st, GK_ERR_INVALID, (unsigned)i);
                u = -1;
            }
            int nq = 0;
            if (u >= 0) {
#pragma unroll
                for (int c = 0; c < KC; c++) {
                    if (32 * c >= kp)
                        break;
                    int v = lab[c];
                    if (v != -3 && (v < 0 || v >= k))
                        flag_error(st, GK_ERR_INVALID, (unsigned)(v == -2 ? i : sg[q * kp + 32 * c + lane]));
                    if (v < 0 || v >= k || v == u)
                        v = -1;
                    bool keep = v >= 0;
#pragma unroll 8
                    for (int z = 0; z < nq; z++)
                        keep &= sq[q * kp + z] != v;
                    const unsigned same = __match_any_sync(FULL_MASK, v);
                    keep = keep && (__ffs(same) - 1 == lane);
                    const unsigned km = __ballot_sync(FULL_MASK, keep);
                    if (keep)
                        sq[q * kp + nq + __popc(km & lanemask_lt())] = v;
                    nq += __popc(km);
                    __syncwarp();
                }
            }
            if (lane == 0) {
                su[q] = u;
                snq[q] = nq;
            }
        }
        __syncthreads();

        // ---- screening: task t of the CTA's visits in turn, B tasks of a warp at once
        const int own_tasks = lane < nv && snq[lane] > 0 ? snq[lane] + 1 : 0;
        int incl = own_tasks;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL_MASK, incl, o);
            if (lane >= o)
                incl += v;
        }
        const int T = __shfl_sync(FULL_MASK, incl, 31), excl = incl - own_tasks;
        for (int t0 = w * B; t0 < T; t0 += BE_WARPS * B) {
            double a[B][PL];
            int ent[B], qb[B];
            double sr = 0.0;
            int nr = 1;
#pragma unroll
            for (int b = 0; b < B; b++) {
                const int t = min(t0 + b, T - 1);
                const int q = __popc(__ballot_sync(FULL_MASK, incl <= t));
                const int c = t - __shfl_sync(FULL_MASK, excl, q);
                const int r = c == 0 ? su[q] : sq[q * kp + c - 1];
                const double *Dr = D + (int64_t)r * d;
                ent[b] = q * ks + c;
                qb[b] = q;
#pragma unroll
                for (int p = 0; p < PL; p++)
                    a[b][p] = lane + 32 * p < d ? __ldcg(Dr + lane + 32 * p) : 0.0;
                if (lane == b) {
                    sr = __ldcg(S + r);
                    nr = __ldcg(cnt + r);
                }
            }
            float dot = 0.f;
            int me = 0, mq = 0;
#pragma unroll
            for (int b = 0; b < B; b++) {
                const float *xq = xs + qb[b] * P;
                float v = 0.f;
#pragma unroll
                for (int p = 0; p < PL; p++)
                    v = fmaf(cut32(a[b][p]), xq[lane + 32 * p], v);
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1)
                    v += __shfl_xor_sync(FULL_MASK, v, o);
                if (lane == b) {
                    dot = v;
                    me = ent[b];
                    mq = qb[b];
                }
            }
            if (lane < B && t0 + lane < T) {
                const float xx = sxx[mq], nf = (float)nr;
                const float rs = sqrtf((float)sr), rx = sqrtf(xx), pr = 1.001f * rs * rx, sn = (float)sr / nf;
                const bool own = me == mq * ks;
                const float den = own ? nf - 1.f : nf + 1.f;
                float g = (own ? xx - 2.f * dot + sn : 2.f * dot + xx - sn) / den;
                float e = ((float)(PL + 16) * 0x1p-23f) * (2.f * pr + xx + sn) / den;
                const bool sure = rs >= 0x1p-40f && rs <= 0x1p60f && rx >= 0x1p-40f && rx <= 0x1p60f &&
                                  nr >= (own ? 2 : 1) && isfinite(g) && isfinite(e);
                tg[me] = sure ? g : 0.f;
                te[me] = sure ? e : __int_as_float(0x7f800000);
                tm[me] = 2.f * (sn + pr + xx);  // no smaller than the terms of the FP64 gain, which round to 2^-44 of it
                en[me] = nr;
                es[me] = sr;
            }
        }
        __syncthreads();
        // ---- the tasks that decide, one warp per visit: none where no gain can be positive.  nev[q]: how many
        //      candidates, or -1 where the only one's gain is positive for sure
        for (int q = w; q < nv; q += BE_WARPS) {
            const int nq = snq[q], o = q * ks;
            int left = 0;
            unsigned in[KC] = {};
            bool sure = false;
            if (nq > 0 && en[o] >= 2) {
                const float inf = __int_as_float(0x7f800000), go = tg[o], eo = te[o], mo = tm[o];
                float low = -inf, g[KC], e[KC];
#pragma unroll
                for (int cc = 0; cc < KC; cc++) {
                    const int c = 1 + 32 * cc + lane;
                    g[cc] = c <= nq ? tg[o + c] : -inf;
                    e[cc] = c <= nq ? te[o + c] + 0x1p-44f * (tm[o + c] + mo) : 0.f;
                    low = fmaxf(low, g[cc] - e[cc]);
                }
#pragma unroll
                for (int h = 16; h >= 1; h >>= 1)
                    low = fmaxf(low, __shfl_xor_sync(FULL_MASK, low, h));
#pragma unroll
                for (int cc = 0; cc < KC; cc++) {
                    const float up = g[cc] + e[cc];
                    const bool may = 1 + 32 * cc + lane <= nq && !(up < low) &&
                                     !(up + go + eo < -1e-6f * (fabsf(up) + fabsf(go)));
                    in[cc] = __ballot_sync(FULL_MASK, may);
                    left += __popc(in[cc]);
                }
                sure = left == 1 && low + go - eo > 1e-6f * (fabsf(low) + fabsf(go));
            }
            int at = 0;
            if (lane == 0) {
                at = left > 0 ? atomicAdd(&s_ne, left + 1) : 0;
                nat[q] = at;
                nev[q] = sure ? -1 : left;
            }
            at = __shfl_sync(FULL_MASK, at, 0);
            if (left > 0) {
                if (lane == 0)
                    tl[at] = o;
                at++;
#pragma unroll
                for (int cc = 0; cc < KC; cc++) {
                    if ((in[cc] >> lane) & 1)
                        tl[at + __popc(in[cc] & lanemask_lt())] = o + 1 + 32 * cc + lane;
                    at += __popc(in[cc]);
                }
            }
        }
        __syncthreads();
        // ---- their squared norms as defined: (D_u - x) for the own cluster, else (D_v + x)
        const int ne = s_ne;
        for (int z = w; z < ne; z += BE_WARPS) {
            const int e = tl[z], q = e / ks, c = e - q * ks;
            const double *Dr = D + (int64_t)(c == 0 ? su[q] : sq[q * kp + c - 1]) * d;
            const float *xq = xs + q * P;
            double a[PL];
#pragma unroll
            for (int p = 0; p < PL; p++)
                a[p] = lane + 32 * p < d ? __ldcg(Dr + lane + 32 * p) : 0.0;
#pragma unroll
            for (int p = 0; p < PL; p++) {
                const double x = widen(xq[lane + 32 * p]);  // on the integer pipe
                const double y = lane + 32 * p < d ? (c == 0 ? __dsub_rn(a[p], x) : __dadd_rn(a[p], x)) : 0.0;
                a[p] = __dmul_rn(y, y);
            }
            const double tot = fold_lanes<PL>(a);
            if (lane == 0)
                ea[e] = tot;
        }
        __syncthreads();
        // ---- each visit's move, written into every CTA of the cluster
        for (int q = w; q < nv; q += BE_WARPS) {
            const int j = q * R + rank, o = q * ks, at = nat[q], left = nev[q];
            int best = left < 0 ? tl[at + 1] : -1;  // the entry of the target
            if (left > 0) {
                // the largest gain, then the smaller label; the gain's integer key orders as its value does (the gains
                // are sums and differences of non-negative terms, never -0); entry 0 of the list is the own cluster
                double r1o = 0.0, r3o = 0.0;
                long long top = LLONG_MIN;
                unsigned long long win = ~0ull;
                for (int z0 = 0; z0 <= left; z0 += 32) {
                    const int z = z0 + lane, e = tl[at + min(z, left)];
                    const double r1 = __ddiv_rn(ea[e], (double)(z == 0 ? en[e] - 1 : en[e] + 1));
                    const double r3 = __ddiv_rn(es[e], (double)en[e]);
                    if (z0 == 0) {
                        r1o = __shfl_sync(FULL_MASK, r1, 0);
                        r3o = __shfl_sync(FULL_MASK, r3, 0);
                    }
                    if (z >= 1 && z <= left) {
                        const double g = __dsub_rn(__dsub_rn(__dadd_rn(r1, r1o), r3), r3o);
                        const long long b = __double_as_longlong(g), key = b ^ ((b >> 63) & 0x7fffffffffffffffll);
                        const unsigned long long id =
                            ((unsigned long long)(unsigned)sq[q * kp + e - o - 1] << 32) | (unsigned)e;
                        if (key > top || (key == top && id < win)) {
                            top = key;
                            win = id;
                        }
                    }
                }
#pragma unroll
                for (int h = 16; h >= 1; h >>= 1) {
                    const long long k2 = __shfl_xor_sync(FULL_MASK, top, h);
                    const unsigned long long w2 = __shfl_xor_sync(FULL_MASK, win, h);
                    if (k2 > top || (k2 == top && w2 < win)) {
                        top = k2;
                        win = w2;
                    }
                }
                if (top > 0)  // the gain is above +0
                    best = (int)(win & 0xffffffffu);
            }
            if (lane < R) {
                st_rank(&mvi[j], lane, svis[q]);
                st_rank(&mvu[j], lane, su[q]);
                st_rank(&mvv[j], lane, best >= 0 ? sq[q * kp + best - o - 1] : -1);
            }
            if (lane == 0)
                mve[q] = best;
        }
        cluster_barrier();

        // ---- the window commits up to the first visit that depends on an earlier moving one: its sample or a neighbour
        //      is that visit's sample, or its own cluster or a candidate is one that visit leaves or joins
        const unsigned moving = __ballot_sync(FULL_MASK, lane < Wn && mvv[min(lane, Wn - 1)] >= 0);
        for (int q = w; q < nv; q += BE_WARPS) {
            const int j = q * R + rank, nq = snq[q], i = svis[q], u = su[q];
            int g[KC], c[KC];
#pragma unroll
            for (int cc = 0; cc < KC; cc++) {
                g[cc] = 32 * cc < kp ? sg[q * kp + 32 * cc + lane] : -1;
                c[cc] = 32 * cc + lane < nq ? sq[q * kp + 32 * cc + lane] : -1;
            }
            bool hit = false;
            for (unsigned left = moving & ((1u << j) - 1u); left; left &= left - 1u) {
                const int b = __ffs(left) - 1, xi = mvi[b], xu = mvu[b], xv = mvv[b];
                hit |= i == xi || u == xu || u == xv;
#pragma unroll
                for (int cc = 0; cc < KC; cc++)
                    hit |= g[cc] == xi || c[cc] == xu || c[cc] == xv;
            }
            hit = __any_sync(FULL_MASK, hit);
            if (lane < R)
                st_rank(&dep[j], lane, hit ? j : Wn);
        }
        cluster_barrier();

        // ---- the committed moves touch disjoint clusters: x leaves D_u for D_v in each, by the CTA that evaluated it
        const int done = (int)__reduce_min_sync(FULL_MASK, (unsigned)(lane < Wn ? dep[lane] : Wn));
        const unsigned commit = moving & (done >= 32 ? ~0u : (1u << done) - 1u);
        moves += __popc(commit);
        for (int z = threadIdx.x; z < nv * d; z += BE_THREADS) {
            const int q = z / d, t = z - q * d, j = q * R + rank;
            if ((commit >> j) & 1u) {
                const double x = widen(xs[q * P + t]);
                double *Du = D + (int64_t)su[q] * d + t, *Dv = D + (int64_t)mvv[j] * d + t;
                const double a = __ldcg(Du), b = __ldcg(Dv);
                *Du = __dsub_rn(a, x);
                *Dv = __dadd_rn(b, x);
            }
        }
        if (threadIdx.x < nv) {
            const int q = threadIdx.x, j = q * R + rank;
            if ((commit >> j) & 1u) {
                const int u = su[q], v = mvv[j], o = q * ks, e = mve[q];
                cnt[u] = en[o] - 1;
                cnt[v] = en[e] + 1;
                S[u] = ea[o];
                S[v] = ea[e];
                L[svis[q]] = v;
            }
        }
        __syncthreads();  // the window's samples are read
        s += done;
        Wn = (int)(m - s < (int64_t)W ? m - s : (int64_t)W);
        cluster_arrive();  // the window's moves before the next window reads labels and rows
        if (s < m)
            fetch(s, Wn);
        cluster_wait();
    }
    if (rank == 0 && threadIdx.x == 0 && n_moved)
        *n_moved = moves;
}

// Largest cluster (at most BE_MAX_CLUSTER CTAs) the device can run for this kernel with `smem` bytes of dynamic
// shared memory per CTA, once per device and kernel.
template <typename KernelT>
int epoch_cluster_size(KernelT kern, size_t smem)
{
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return 0;
    std::lock_guard<std::mutex> lock(mu);
    auto key = std::make_pair(dev, reinterpret_cast<const void *>(kern));
    auto it = known.find(key);
    if (it != known.end())
        return it->second;
    int r = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess) {
        r = 8;  // portable size
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(BE_MAX_CLUSTER);
            cfg.blockDim = dim3(BE_THREADS);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = BE_MAX_CLUSTER;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int most = 0;
            if (cudaOccupancyMaxPotentialClusterSize(&most, kern, &cfg) == cudaSuccess && most > 0)
                r = most < BE_MAX_CLUSTER ? most : BE_MAX_CLUSTER;
        }
    }
    cudaGetLastError();
    known[key] = r;
    return r;
}

template <typename XT, int PL>
cudaError_t boost_epoch_t(const XT *X, int64_t n, int64_t d, int64_t ld, const int32_t *G, int32_t kappa,
                          const int32_t *order, int64_t m, int32_t *L, int32_t k, double *D, int32_t *cnt, double *S,
                          int64_t *n_moved, DevStatus *st, cudaStream_t s)
{
    auto kern = k_boost_epoch<XT, PL>;
    const int R = epoch_cluster_size(kern, BE_SMEM_BUDGET);
    if (R < 1)
        return cudaErrorInvalidConfiguration;
    int W = BE_MAX_WINDOW;  // the largest window whose layout fits the budget
    while (W > 1 && WinLayout(W, 32 * PL, kappa, R).bytes > BE_SMEM_BUDGET)
        W--;
    const size_t smem = WinLayout(W, 32 * PL, kappa, R).bytes;
    if (smem > BE_SMEM_BUDGET)
        return cudaErrorInvalidConfiguration;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)R);
    cfg.blockDim = dim3(BE_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)R;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, X, (int32_t)n, (int)d, ld, G, (int)kappa, order, m, L, k, D, cnt, S,
                              n_moved, st, W);
}

template <int PL>
cudaError_t boost_epoch_pl(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *G, int32_t kappa,
                           const int32_t *order, int64_t m, int32_t *L, int32_t k, double *D, int32_t *cnt, double *S,
                           int64_t *n_moved, DevStatus *st, cudaStream_t s)
{
    if (bf16)
        return boost_epoch_t<__nv_bfloat16, PL>(static_cast<const __nv_bfloat16 *>(X), n, d, ld, G, kappa, order, m, L,
                                                k, D, cnt, S, n_moved, st, s);
    return boost_epoch_t<float, PL>(static_cast<const float *>(X), n, d, ld, G, kappa, order, m, L, k, D, cnt, S,
                                    n_moved, st, s);
}

template <int PL>
cudaError_t boost_norms_pl(const double *D, int64_t d, int32_t k, const int32_t *offsets, double *S, int32_t *counts,
                           cudaStream_t s)
{
    k_boost_norms<PL><<<(k + 7) / 8, 256, 0, s>>>(D, (int)d, k, offsets, S, counts);
    return cudaGetLastError();
}

int lanes_per_row(int64_t d)
{
    int pl = 1;
    while (32 * pl < d)
        pl <<= 1;
    return pl;
}

}  // namespace

int64_t boost_max_d() { return BO_MAX_D; }

cudaError_t launch_boost_init(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *labels,
                              int32_t k, double *D, int32_t *counts, double *S, int32_t *offsets, int32_t *members,
                              int32_t *grp_counts, void *grp_scratch, DevStatus *st, cudaStream_t s)
{
    cudaError_t e = launch_group(labels, n, k, offsets, members, grp_counts, grp_scratch, st, s);
    if (e != cudaSuccess)
        return e;
    const dim3 grid((unsigned)k, (unsigned)((d + BS_THREADS - 1) / BS_THREADS));
    if (bf16)
        k_boost_sum<__nv_bfloat16><<<grid, BS_THREADS, 0, s>>>(static_cast<const __nv_bfloat16 *>(X), (int)d, ld,
                                                               offsets, members, D);
    else
        k_boost_sum<float><<<grid, BS_THREADS, 0, s>>>(static_cast<const float *>(X), (int)d, ld, offsets, members, D);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    switch (lanes_per_row(d)) {
    case 1: return boost_norms_pl<1>(D, d, k, offsets, S, counts, s);
    case 2: return boost_norms_pl<2>(D, d, k, offsets, S, counts, s);
    case 4: return boost_norms_pl<4>(D, d, k, offsets, S, counts, s);
    case 8: return boost_norms_pl<8>(D, d, k, offsets, S, counts, s);
    case 16: return boost_norms_pl<16>(D, d, k, offsets, S, counts, s);
    default: return boost_norms_pl<32>(D, d, k, offsets, S, counts, s);
    }
}

cudaError_t launch_boost_epoch(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *G,
                               int32_t kappa, const int32_t *order, int64_t m, int32_t *labels, int32_t k, double *D,
                               int32_t *counts, double *S, int64_t *n_moved, DevStatus *st, cudaStream_t s)
{
    switch (lanes_per_row(d)) {
    case 1: return boost_epoch_pl<1>(X, bf16, n, d, ld, G, kappa, order, m, labels, k, D, counts, S, n_moved, st, s);
    case 2: return boost_epoch_pl<2>(X, bf16, n, d, ld, G, kappa, order, m, labels, k, D, counts, S, n_moved, st, s);
    case 4: return boost_epoch_pl<4>(X, bf16, n, d, ld, G, kappa, order, m, labels, k, D, counts, S, n_moved, st, s);
    case 8: return boost_epoch_pl<8>(X, bf16, n, d, ld, G, kappa, order, m, labels, k, D, counts, S, n_moved, st, s);
    case 16: return boost_epoch_pl<16>(X, bf16, n, d, ld, G, kappa, order, m, labels, k, D, counts, S, n_moved, st, s);
    default: return boost_epoch_pl<32>(X, bf16, n, d, ld, G, kappa, order, m, labels, k, D, counts, S, n_moved, st, s);
    }
}

}  // namespace gkm
