// Block products on row-classed entries and packed rows of X (block.cu).
#pragma once

#include "ff_internal.cuh"

namespace ff {

struct BlockPlan;

// The block layout of A (or A^T), built on first use from the handle's host
// copy of the matrix (synchronous, one allocation); null while `st` is being
// captured into a graph before that, or when the layout cannot be made (2^32
// entries, no memory): the caller then takes the plan's own path.
const BlockPlan *ensure_block(ffspmv_handle *h, bool transpose, cudaStream_t st);
void free_block(ffspmv_handle *h);
long long block_launches(const BlockPlan &B, int nvec);  // of a contiguous, 16-byte aligned block
ffspmv_status run_block(const BlockPlan &B, const u32 *x, long long ldx, u32 *y, long long ldy, int nvec, u32 m,
                        u32 alpha, u32 beta, cudaStream_t st);

// Y_j = A_j X_j of different plans, one product launch per 512 of them:
// contiguous blocks of nvec[j] <= 32 vectors.
ffspmv_status run_block_many(int count, const BlockPlan *const *B, const u32 *const *x, u32 *const *y, const int *nvec,
                             cudaStream_t st);

}  // namespace ff
