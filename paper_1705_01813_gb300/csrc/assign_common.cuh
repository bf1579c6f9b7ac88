// Helpers shared by the assignment kernels (SIMT and tensor-core): the
// per-lane partial squared distance in the fixed order of the FP32 path and
// the warp reductions that complete it.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace gkm {

// Warp sums of G per-lane partial values (G = 2, 4, ..., 32 candidates) at
// once.  The first log2 G exchange steps pair lanes across bit 4, 3, ... and
// halve the values each lane holds; the remaining lane bits are summed with a
// plain xor butterfly.  Every candidate's total is thus formed with the tree
// of warp_total (bit 4 first, then 3, 2, 1, 0), so all three give the same
// bits.  Afterwards lane l holds the total of candidate l / (32 / G).
// With LPR = 8 or 16 the lanes of each LPR have their own G candidates: rows
// of at most LPR vectors leave the lanes from LPR on at +0 in warp_total's
// tree, which adds nothing, so the totals are that tree's here too (lane l of
// the LPR holds candidate l / (LPR / G)).
template <int G, int LPR = 32>
__device__ __forceinline__ float transpose_reduce(float (&v)[G])
{
    static_assert(G >= 2 && G <= LPR && (G & (G - 1)) == 0, "G must be a power of two in [2, LPR]");
    const int lane = lane_id();
#pragma unroll
    for (int h = G / 2, o = LPR / 2; h >= 1; h >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < h; j++) {
            float send = upper ? v[j] : v[j + h];
            float keep = upper ? v[j + h] : v[j];
            v[j] = keep + __shfl_xor_sync(FULL_MASK, send, o);
        }
    }
    float t = v[0];
#pragma unroll
    for (int o = LPR / 2 / G; o >= 1; o >>= 1)
        t += __shfl_xor_sync(FULL_MASK, t, o);
    return t;
}

__device__ __forceinline__ float transpose_reduce32(float (&v)[32]) { return transpose_reduce<32>(v); }

// Partial (per lane) squared distance of x (registers) to a row of 16-byte
// vectors, in the accumulation order of the assignment kernels: two
// accumulators, (a0, a1) += (e0^2, e1^2), then += (e2^2, e3^2) per vector,
// each a round-to-nearest FMA, and a0 + a1 at the end.  The packed FP32x2 FMA
// of sm_100+ performs each pair at once with the same roundings; e = x - c is
// formed as fma(c, -1, x), which is x - c rounded once.
template <int NV, int LPR = 32, typename RowLoad>
__device__ __forceinline__ float lane_partial(const float4 (&xv)[NV], int d4, RowLoad load)
{
    const int lane = LPR == 32 ? lane_id() : lane_id() & (LPR - 1);
    const float2 m1 = make_float2(-1.f, -1.f);
    float2 a = make_float2(0.f, 0.f);
#pragma unroll
    for (int v = 0; v < NV; v++) {
        const int col = lane + 32 * v;
        if (col < d4) {
            const float4 cv = load(col);
            const float2 e01 = __ffma2_rn(make_float2(cv.x, cv.y), m1, make_float2(xv[v].x, xv[v].y));
            const float2 e23 = __ffma2_rn(make_float2(cv.z, cv.w), m1, make_float2(xv[v].z, xv[v].w));
            a = __ffma2_rn(e01, e01, a);
            a = __ffma2_rn(e23, e23, a);
        }
    }
    return a.x + a.y;
}

// Complete one candidate's distance from the lane partials: the xor butterfly
// pairs lanes by bit 4, then 3, 2, 1, 0, which is the grouping of
// transpose_reduce32, so the total has the same bits as there.
__device__ __forceinline__ float warp_total(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

}  // namespace gkm
