// Block products on row-classed entries and packed rows of X (block.cu).
#pragma once

#include "ff_internal.cuh"

namespace ff {

constexpr int kBlockThreads = 256;
constexpr long long kBlockLong = 512;   // entries of a chunk; longer rows are split over warps
constexpr int kBlockVecs = 32;          // vectors per pass
constexpr int kBlockClasses = 7;        // by quads of entries: 0, 1, 2, 3-4, 5-8, 9-16, 17-128

// log2 of the groups per row of class i (heaviest first), 2^lgt lanes per row
// of X.  A group's epilogue (sums joined, one reduction per component) costs
// about as much as three quads, so rows share as few groups as keep the warp's
// lanes busy: with four or more lanes per row of X fewer still.  300 007 x
// 200 003, 22 per row, m = 2^31 - 1, 16 vectors: 79 us with 8 / 4 / 2 groups
// for classes 1 to 3, 59 with 4 / 2 / 1, 53 with 2 / 1 / 1 (3 vectors: 39, 39,
// 45).
__host__ __device__ inline int block_lgg(int i, int lgt)
{
    const int lg = i == 0 ? 4 : lgt < 2 ? (i == 1 ? 2 : i == 2 ? 1 : 0) : i == 1 ? 1 : 0;
    return lg < 5 - lgt ? lg : 5 - lgt;
}

struct BlockDev;   // what a launch over many matrices reads of each (block.cu)

constexpr int kBlockStagings = 7;       // of 1, 2, 4, ... 16-byte pieces per row of X: up to 8 for a block,
constexpr int kBlockPieces = 1 << (kBlockStagings - 1);   // ... more for several blocks of a batch

// When to ask again for device memory that was not there: after 1, 2, 4, ...
// (at most 1024) more calls.
struct BlockMemory {
    bool short_of = false;
    int calls = 0, wait = 1;
    bool again() { return short_of && ++calls >= wait; }
    void next(const BlockMemory &before)   // asked again, in vain if short_of
    {
        calls = 0;
        wait = before.wait < 1024 ? 2 * before.wait : before.wait;
    }
};

struct BlockPlan {
    bool ok = false;
    BlockMemory memory, staging;
    const BlockDev *dev = nullptr;
    void *arena = nullptr;
    long long n = 0, ncols = 0;
    bool small = true;                 // m <= 2^16: u16 values and staged x
    int nsm = 1;                       // the device's SMs
    long long nlong = 0, nchunk = 0;   // rows split over warps, and their chunks
    long long cls_row[kBlockClasses + 1] = {};  // rows of class c: [cls_row[c], cls_row[c + 1]) of row / ptr
    const u32 *ptr = nullptr;          // [n - nlong + 1] offsets in quads, rows in class order
    const u32 *row = nullptr;          // [n - nlong] their matrix rows
    const uint4 *chunk = nullptr;      // (long row index, first quad, end, chunks of the row)
    const u32 *lrow = nullptr;         // [nlong] matrix rows
    const u32 *col = nullptr;
    const void *val = nullptr;
    // Packed rows of X: buffer k holds rows of up to 2^k pieces.  Each is made
    // for the first block that needs it and kept (a captured graph may name it):
    // buffer lgx with the layout, in its allocation.
    uint4 *xs[kBlockStagings] = {};
    int lgx = -1;
    u32 quad1 = 0;                     // the one-quad class: row r at quad quad1 + r (mod 2^32)
    u64 *carry = nullptr;              // [nlong][kBlockVecs], zero between calls
    u32 *count = nullptr;              // [nlong][kBlockVecs] chunks arrived, zero between calls
};

// A block layout of A or A^T, made on the device (synchronous); `odd`: of the
// pattern of the odd values, padded with columns 2^32 - 1, without values and
// without sums of long rows; lgx: with packed rows of 2^lgx pieces (-1: none).  On
// an error other than a stream under capture or no host memory *out is a plan
// with ok = false.
ffspmv_status make_block(const ffspmv_handle *h, bool transpose, bool odd, int lgx, cudaStream_t st, BlockPlan **out);
void free_block_plan(BlockPlan *b);

// The block layout of A (or A^T), built on first use from the handle's host
// copy of the matrix (synchronous, one allocation); null while `st` is being
// captured into a graph before that, or when the layout cannot be made (2^32
// entries; no memory, which is asked for again later): the caller then takes
// the plan's own path.  A new layout comes with the staging for the block x (nvec
// = 0: none).
BlockPlan *ensure_block(ffspmv_handle *h, bool transpose, const u32 *x, long long ldx, int nvec, cudaStream_t st);
// The same for the A of several different handles, before a batch of contiguous
// blocks: what is missing is built together.
void ensure_blocks(int count, ffspmv_handle *const *hs, const u32 *const *x, const int *nvec, cudaStream_t st);
void free_block(ffspmv_handle *h);
void block_handles(int more);   // a handle was made (1) or freed (-1)
std::string block_summary(const BlockPlan *b);   // a line of spmv_describe_plan
// The buffer for the packed rows of a block (null where all its rows are read
// in place), allocated for the first block of that width.  False when it is not
// there and cannot be made now (a capture, no memory): the plan's own path.
bool block_staging(BlockPlan &B, const u32 *x, long long ldx, int nvec, cudaStream_t st, uint4 **xs);
long long block_launches(const BlockPlan &B, int nvec);  // of a contiguous, 16-byte aligned block
ffspmv_status run_block(const BlockPlan &B, uint4 *xs, const u32 *x, long long ldx, u32 *y, long long ldy, int nvec,
                        u32 m, u32 alpha, u32 beta, cudaStream_t st);

// Pieces per packed row of a contiguous block; 0 where it is read in place.
int block_pieces(const BlockPlan &B, const u32 *x, int nvec);
// A staging buffer for several blocks of one plan at a time, of at most `most`
// pieces each and `total` in all: with room for *room pieces, as many as up to
// kBlockPieces and 64 MB allow (null: not there and cannot be made now).
uint4 *block_staging(BlockPlan &B, int most, int total, cudaStream_t st, int *room);

// Y_j = A_j X_j, one product launch per 512 of them: contiguous blocks of nvec[j]
// <= 32 vectors, each with its staging.  Blocks of one plan need stagings of
// their own and, where it has long rows, words v0[j] .. v0[j] + nvec[j] - 1 of 32.
ffspmv_status run_block_many(int count, const BlockPlan *const *B, uint4 *const *xs, const u32 *const *x, u32 *const *y,
                             const int *nvec, const int *v0, cudaStream_t st);

// nsteps >= 1 steps of a block sequence at m > 2^16, one launch each and one
// more: S_i = X^T V_i (at S + i s s) and V_{i+1} = A V_i between V0 and V1 (n
// rows of s words rounded up to 4, zero past s; V_0 in V0; `next`: V_nsteps is
// formed too).  part: block_steps_bytes of scratch.
size_t block_steps_bytes(long long n, int s);
ffspmv_status run_block_steps(const BlockPlan &B, long long n, int s, u32 m, const u32 *X, u32 *V0, u32 *V1, u32 *part,
                              long long nsteps, bool next, u32 *S, cudaStream_t st);

}  // namespace ff
