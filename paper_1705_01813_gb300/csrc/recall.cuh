// Tensor-core screening of the recall estimator's queries (recall_tc.cu), used by recall.cu.
#pragma once

#include "common.cuh"

namespace gkm {

size_t recall_screen_bytes(int64_t d, int32_t m);
// best[q]: the smallest (distance, id) key of query q among the other samples; the *nleft queries (indexes in *left,
// both on the device) that the screening leaves to the FP32 tiles keep what best held.
cudaError_t launch_recall_screen(const void *X, bool bf16, int64_t n, int64_t d, int64_t ld, const int32_t *g_idx,
                                 int32_t kappa, const int32_t *queries, int32_t m, uint64_t *best, void *scratch,
                                 const int32_t **left, const int32_t **nleft, DevStatus *st, cudaStream_t s);

}  // namespace gkm
