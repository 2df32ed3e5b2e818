// Polynomial-matrix products inside the library (polymat.cu): rectangular
// operands and windows of the product, as the sigma-basis recursion uses them.
#pragma once

#include "ff_internal.cuh"

namespace ff {

// Node of the sigma-basis recursion on the device: shifted degrees delta of
// its basis, the bound e on its degree, the largest delta and the least input
// shift.
struct SbSlot {
    int e, smin, dmax;
    int bad;             // a bounded wait of a leaf below ran out
    int delta[32];
};

// Workspace (bytes) of pm_product for these sizes, or 0 when the transform
// would be too long.
size_t pm_product_bytes(int sr, int si, int sc, long long da, long long db, long long klo, long long khi, int npr = 3);

// C = the coefficients klo..khi of A(x) B(x) mod p, through transforms: A has
// da + 1 coefficients of sr x si, B db + 1 of si x sc (residues below p), C
// khi - klo + 1 of sr x sc; khi <= da + db.
ffspmv_status pm_product(u32 p, int sr, int si, int sc, long long da, long long db, const u32 *A, const u32 *B, u32 *C,
                         long long klo, long long khi, void *work, size_t work_bytes, cudaStream_t st);

// The same by the definition, for short operands, one launch: coefficients of
// A above *ea and of B above *eb (device words, may be null: da and db) are
// taken as zero, so khi may exceed their degrees.  With `out`, the launch
// also forms the node of the product B2 B1: out->e = min(d, s1->e + s2->e,
// s2->dmax - s1->smin) or, when `leaf`, min(d, s2->dmax - s1->smin).
struct PmNode {
    const SbSlot *s1, *s2;
    SbSlot *out;
    int d, leaf, m;
};
// Threads 0..31 of one warp.
__device__ __forceinline__ void pm_node(const PmNode &n, int t)
{
    if (t < n.m) n.out->delta[t] = n.s2->delta[t];
    if (t == 0) {
        int e = min(n.d, n.s2->dmax - n.s1->smin);
        if (!n.leaf) e = min(e, n.s1->e + n.s2->e);
        n.out->e = max(0, e);
        n.out->smin = n.s1->smin;
        n.out->dmax = n.s2->dmax;
        n.out->bad = n.s1->bad | n.s2->bad;
    }
}

ffspmv_status pm_direct(u32 p, int sr, int si, int sc, int da, int db, const u32 *A, const u32 *B, u32 *C, int klo,
                        int khi, const int *ea, const int *eb, const PmNode *node, cudaStream_t st);

}  // namespace ff
