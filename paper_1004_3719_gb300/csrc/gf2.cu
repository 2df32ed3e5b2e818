// Products over GF(2) = Z/2Z with bit-packed vectors: Y = A X or A^T X (or
// Y ^= ...), X holding 64 components per 64-bit word.  This is Sec. 2's
// y_i = sum_j A_ij x_j at m = 2, where a sum is an exclusive or and an entry
// counts when its value is odd; packing the components of a block of vectors
// into words is the binary case the paper's closing remarks point to.
//
// Only the pattern of the odd entries is kept (built on the first call, for A
// or A^T), in the block layout (block.cu): rows in length classes, columns in
// quads, so that a lane loads four columns at once and has four gathers in
// flight while the next quad is on its way.  A lane gathers one 64-bit word of
// a row of X, or two where the rows are 16-byte aligned; T lanes take a row's
// words and G groups of them share a row of A.  The chunks of a row above 512
// entries meet in Y by atomic exclusive or: a launch before clears those rows
// (unless accumulating), and only the chunks' last step waits for it.  Nothing
// of the handle is written, so calls on one handle may overlap.
//
// The gathers bound it: one random L2 sector per entry, 63 us for 15.8M at 250 G
// sectors/s.  1M power-law pattern, 64 / 256 vectors: 91 / 211 us with a lane
// group per short row, a second launch for the long rows and 8-byte offsets;
// 66 / 82 us here (16 words: 1359 -> 302).
#include <algorithm>

#include "ff_block.h"
#include "ff_internal.cuh"

namespace ff {

void free_gf2(ffspmv_handle *h)
{
    for (BlockPlan *&g : h->gf2) {
        free_block_plan(g);
        g = nullptr;
    }
}

namespace {

constexpr int kGf2Lanes = 8;   // lanes per row of X in one pass

struct Gf2Args {
    const u32 *ptr, *row, *col, *lrow;
    const uint4 *chunk;
    const u64 *X;
    u64 *Y;
    int w, pieces, lgt, accumulate;   // words per row of X and Y; pieces of this pass; log2 of the lanes that take them
    u32 nchunk;
    u32 quad1;
    u32 warp0[kBlockClasses + 1], row0[kBlockClasses + 1];
    int lgg[kBlockClasses];
};

// One piece of a row of X: E 64-bit words.
template <int E>
struct Gf2Piece;
template <>
struct Gf2Piece<1> {
    u64 a;
    __device__ __forceinline__ void zero() { a = 0; }
    __device__ __forceinline__ void load(const u64 *p) { a = __ldg(p); }
    __device__ __forceinline__ void add(const Gf2Piece &o) { a ^= o.a; }
    __device__ __forceinline__ void shfl(int off) { a ^= __shfl_xor_sync(0xffffffffu, a, off); }
    __device__ __forceinline__ u64 get(int) const { return a; }
};
template <>
struct Gf2Piece<2> {
    u64 a, b;
    __device__ __forceinline__ void zero() { a = b = 0; }
    __device__ __forceinline__ void load(const u64 *p)
    {
        const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(p));
        a = v.x;
        b = v.y;
    }
    __device__ __forceinline__ void add(const Gf2Piece &o)
    {
        a ^= o.a;
        b ^= o.b;
    }
    __device__ __forceinline__ void shfl(int off)
    {
        a ^= __shfl_xor_sync(0xffffffffu, a, off);
        b ^= __shfl_xor_sync(0xffffffffu, b, off);
    }
    __device__ __forceinline__ u64 get(int i) const { return i ? b : a; }
};

// exclusive or of the pieces that quads k, k + step, ... below end name
template <int E>
__device__ __forceinline__ void gf2_quads(Gf2Piece<E> &acc, const Gf2Args &a, u32 k, u32 end, u32 step, const u64 *xb, bool on)
{
    constexpr u32 kNone = 0xffffffffu;
    uint4 j = make_uint4(kNone, kNone, kNone, kNone);
    if (k < end) j = __ldcs(reinterpret_cast<const uint4 *>(a.col) + k);
    while (k < end) {
        Gf2Piece<E> x[4];
        const u32 c[4] = {j.x, j.y, j.z, j.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[u].zero();
            if (on && c[u] != kNone) x[u].load(xb + (u64)c[u] * (u32)a.w);
        }
        k += step;
        if (k < end) j = __ldcs(reinterpret_cast<const uint4 *>(a.col) + k);
        x[0].add(x[1]);
        x[2].add(x[3]);
        x[0].add(x[2]);
        acc.add(x[0]);
    }
}

// The rows of Y that chunks add to.
__global__ void __launch_bounds__(kBlockThreads) k_gf2_clear(const u32 *__restrict__ lrow, u32 nlong, int w, u64 *Y)
{
    asm volatile("griddepcontrol.launch_dependents;");
    const u64 n = (u64)nlong * (u32)w, step = (u64)gridDim.x * kBlockThreads;
    for (u64 t = (u64)blockIdx.x * kBlockThreads + threadIdx.x; t < n; t += step)
        Y[(size_t)__ldg(lrow + t / (u32)w) * w + t % (u32)w] = 0;
}

// One warp per chunk of a long row, or per 32 / (T G) rows of a class.
template <int E>
__global__ void __launch_bounds__(kBlockThreads) k_gf2(const __grid_constant__ Gf2Args a)
{
    const u32 w = blockIdx.x * (kBlockThreads / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31, T = 1 << a.lgt, c = lane & (T - 1);
    const bool on = c < a.pieces;
    const u64 *xb = a.X + E * c;
    Gf2Piece<E> acc;
    acc.zero();
    if (w < a.nchunk) {
        const uint4 ch = __ldg(a.chunk + w);
        gf2_quads<E>(acc, a, ch.y + (u32)(lane >> a.lgt), ch.z, 32u >> a.lgt, xb, on);
        for (int off = T; off < 32; off <<= 1) acc.shfl(off);
        asm volatile("griddepcontrol.wait;" ::: "memory");   // the row is cleared
        if (lane < T && on) {
            u64 *yp = a.Y + (size_t)__ldg(a.lrow + ch.x) * a.w + E * c;
#pragma unroll
            for (int i = 0; i < E; ++i)
                atomicXor(reinterpret_cast<unsigned long long *>(yp + i), (unsigned long long)acc.get(i));
        }
        return;
    }
    int b = 0;
#pragma unroll
    for (int i = 1; i < kBlockClasses; ++i)
        if (w >= a.warp0[i]) b = i;
    if (w >= a.warp0[kBlockClasses]) return;
    const int lgg = a.lgg[b], lgr = a.lgt + lgg;
    const u64 r64 = a.row0[b] + ((u64)(w - a.warp0[b]) << (5 - lgr)) + (u64)(lane >> lgr);
    const bool ok = r64 < a.row0[b + 1];
    const u32 r = (u32)r64;
    u32 s = 0, e = 0, row = 0;
    if (ok) {
        const bool one = b == kBlockClasses - 2;
        s = one ? a.quad1 + r : __ldg(a.ptr + r);
        e = one ? s + 1u : __ldg(a.ptr + r + 1);
        row = __ldg(a.row + r);
    }
    gf2_quads<E>(acc, a, s + (u32)((lane >> a.lgt) & ((1 << lgg) - 1)), e, 1u << lgg, xb, on);
    for (int off = T; off < 1 << lgr; off <<= 1) acc.shfl(off);
    if (ok && on && (lane & ((1 << lgr) - 1)) < T) {
        u64 *yp = a.Y + (size_t)row * a.w + E * c;
#pragma unroll
        for (int i = 0; i < E; ++i) yp[i] = a.accumulate ? yp[i] ^ acc.get(i) : acc.get(i);
    }
}

}  // namespace
}  // namespace ff

using namespace ff;

extern "C" ffspmv_status spmv_apply_gf2(ffspmv_t h, int32_t transpose, const uint64_t *d_X, uint64_t *d_Y,
                                        int32_t words, int32_t accumulate, ffspmv_stream_t stream)
{
    if (!h || words < 1 || (transpose != 0 && transpose != 1)) return FFSPMV_ERR_ARG;
    if (h->m != 2u) return FFSPMV_ERR_UNSUPPORTED;
    const long long in_rows = transpose ? h->A.nrows : h->A.ncols;
    const long long out_rows = transpose ? h->A.ncols : h->A.nrows;
    if ((in_rows > 0 && !d_X) || (out_rows > 0 && !d_Y)) return FFSPMV_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (!h->gf2[transpose]) {
        BlockPlan *g = nullptr;
        const ffspmv_status r = make_block(h, transpose != 0, true, -1, st, &g);
        if (r != FFSPMV_OK) {
            free_block_plan(g);
            return r;
        }
        h->gf2[transpose] = g;
    }
    const BlockPlan &B = *h->gf2[transpose];
    if (out_rows == 0) return FFSPMV_OK;
    const bool clear = !accumulate && B.nchunk > 0;
    if (clear) {
        const long long n = B.nlong * words;
        k_gf2_clear<<<(unsigned)std::min<long long>((n + kBlockThreads - 1) / kBlockThreads, 4096), kBlockThreads, 0, st>>>(
            B.lrow, (u32)B.nlong, words, (u64 *)d_Y);
        FF_CUDA(cudaGetLastError());
    }
    // two words per lane where every row of X starts on 16 bytes
    const int E = words % 2 == 0 && ((uintptr_t)d_X & 15u) == 0 ? 2 : 1;
    for (int w0 = 0; w0 < words; w0 += E * kGf2Lanes) {
        Gf2Args a;
        memset(&a, 0, sizeof(a));
        a.ptr = B.ptr;
        a.row = B.row;
        a.col = B.col;
        a.lrow = B.lrow;
        a.chunk = B.chunk;
        a.quad1 = B.quad1;
        a.X = (const u64 *)d_X + w0;
        a.Y = (u64 *)d_Y + w0;
        a.w = words;
        a.pieces = std::min(kGf2Lanes, (words - w0) / E);
        while ((1 << a.lgt) < a.pieces) ++a.lgt;
        a.accumulate = accumulate ? 1 : 0;
        a.nchunk = (u32)B.nchunk;
        long long warps = B.nchunk;
        for (int c = 0; c < kBlockClasses; ++c) {
            a.lgg[c] = block_lgg(c, a.lgt);
            a.row0[c] = (u32)B.cls_row[c];
            a.warp0[c] = (u32)warps;
            const int rpw = 32 >> (a.lgt + a.lgg[c]);
            warps += (B.cls_row[c + 1] - B.cls_row[c] + rpw - 1) / rpw;
        }
        a.row0[kBlockClasses] = (u32)B.cls_row[kBlockClasses];
        a.warp0[kBlockClasses] = (u32)warps;
        if (warps >= (1LL << 32) - 1) return FFSPMV_ERR_UNSUPPORTED;
        // the first pass starts while the rows are cleared
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((warps * 32 + kBlockThreads - 1) / kBlockThreads));
        cfg.blockDim = dim3(kBlockThreads);
        cfg.stream = st;
        cfg.attrs = &attr;
        cfg.numAttrs = clear && w0 == 0 ? 1 : 0;
        FF_CUDA(cudaLaunchKernelEx(&cfg, E == 2 ? k_gf2<2> : k_gf2<1>, a));
    }
    return FFSPMV_OK;
}
