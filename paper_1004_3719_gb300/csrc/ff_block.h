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

// nsteps >= 1 steps of a block sequence at m > 2^16, one launch each and one
// more: S_i = X^T V_i (at S + i s s) and V_{i+1} = A V_i between V0 and V1 (n
// rows of s words rounded up to 4, zero past s; V_0 in V0; `next`: V_nsteps is
// formed too).  part: block_steps_bytes of scratch.
size_t block_steps_bytes(long long n, int s);
ffspmv_status run_block_steps(const BlockPlan &B, long long n, int s, u32 m, const u32 *X, u32 *V0, u32 *V1, u32 *part,
                              long long nsteps, bool next, u32 *S, cudaStream_t st);

}  // namespace ff
