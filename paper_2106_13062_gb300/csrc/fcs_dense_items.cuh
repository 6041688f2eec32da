// fcs_dense_items.cuh -- host interface of fcs_dense_items.cu.
#pragma once

#include "fcs_internal.cuh"

namespace fcs {

// Issues the dense sketch of a batch of small, densely packed tensors and sets
// *done when the shape is one for it; otherwise nothing is issued.  off[n]:
// offset of mode n in a hash-table row.
int dense_items(fcs_ctx *ctx, int N, const int64_t *I, const int64_t *stride, const int64_t *off,
                const int32_t *J, int64_t ldh, int64_t Jt, int D, const float *T, const int32_t *h,
                const int8_t *s, float *out, int64_t nbatch, int64_t tbs, int64_t obs, bool *done);

}  // namespace fcs
