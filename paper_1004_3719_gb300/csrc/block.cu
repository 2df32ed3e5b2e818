// Y <- alpha A X + beta Y for blocks of vectors (Sec. 2.5.1): one pass over
// the matrix for up to 32 vectors.
//
// A gather of x costs one 32-byte L2 sector however little of it is used, and
// the gathers are what bounds a row-wise product (about 250 G sectors/s
// measured on this chip).  With the residues of one row of X packed next to
// each other (u16 for m <= 2^16: 16 vectors are 32 bytes), one sector serves
// all the vectors, so a pass takes about the time of one vector's gathers.
// The x-panel layout, which is faster for one vector, has no such gain: its
// panels and row groups shrink as x and the row sums widen.  Measured on the
// 1M x 1M power-law matrix (15.8M entries, m = 65521), 16 vectors: 643 us
// in passes of the x-panel layout, 128 us here (14 us of it the packing); 16
// vectors at m = 2^31 - 1: 1093 -> 181 us; 90 001 x 120 011 with power-law rows
// (binned plan): 515 -> 20 us.
//
// Layout.  Rows are ordered by length class and their entries stored in that
// order, so that the lanes of a warp do the same number of steps; T lanes
// hold the 16-byte pieces of a row of X (T = 1, 2, 4, 8), G groups of T lanes
// share a matrix row (G grows with the class).  Rows above kBlockLong entries
// are cut into chunks of that many, one warp each; the chunks add reduced
// sums into 64-bit words and the last one to arrive writes the row.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <exception>
#include <mutex>
#include <new>
#include <string>
#include <thread>
#include <type_traits>

#include "ff_internal.cuh"
#include "ff_block.h"

namespace ff {
namespace {

__device__ __forceinline__ int block_class(u32 quads)
{
    return quads <= 2u ? (int)quads : min(kBlockClasses - 1, 33 - __clz(quads - 1u));
}

}  // namespace

// What a launch over many matrices reads of each (k_block_many).
struct BlockDev {
    const u32 *ptr, *row, *col, *lrow;
    const uint4 *chunk;
    const void *val;
    u64 *carry;
    u32 *count;
    long long ncols;
    u32 row0[kBlockClasses + 1];  // rows of each class, heaviest class first
    u32 nchunk, quad1;
    int small, fold;
    Mod M;
};

void free_block(ffspmv_handle *h)
{
    for (BlockPlan *&b : h->block) {
        free_block_plan(b);
        b = nullptr;
    }
}

namespace {

// Word t of the rows of X packed to `pitch` 16-byte words each: u16 or u32
// residues, zero past nvec.
template <bool SMALL>
__device__ __forceinline__ uint4 block_pack(const u32 *__restrict__ x, long long ldx, long long t, int nvec, int pitch, int vec4)
{
    constexpr int C = SMALL ? 8 : 4;
    const long long i = t / pitch;
    const int c0 = (int)(t - i * pitch) * C;
    const u32 *p = x + i * ldx + c0;
    u32 v[C];
    if (vec4 && c0 + C <= nvec) {
#pragma unroll
        for (int u = 0; u < C / 4; ++u) {
            const uint4 w = __ldg(reinterpret_cast<const uint4 *>(p) + u);
            v[4 * u] = w.x; v[4 * u + 1] = w.y; v[4 * u + 2] = w.z; v[4 * u + 3] = w.w;
        }
    } else {
#pragma unroll
        for (int u = 0; u < C; ++u) v[u] = c0 + u < nvec ? __ldg(p + u) : 0u;
    }
    if constexpr (SMALL)
        return make_uint4((v[0] & 0xffffu) | v[1] << 16, (v[2] & 0xffffu) | v[3] << 16, (v[4] & 0xffffu) | v[5] << 16,
                          (v[6] & 0xffffu) | v[7] << 16);
    else
        return make_uint4(v[0], v[1], v[2], v[3]);
}

template <bool SMALL>
__global__ void __launch_bounds__(kBlockThreads) k_block_stage(const u32 *__restrict__ x, long long ldx, long long n,
                                                              int nvec, int pitch, int vec4, uint4 *__restrict__ xs)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t = (long long)blockIdx.x * kBlockThreads + threadIdx.x;
    if (t < n * pitch) xs[t] = block_pack<SMALL>(x, ldx, t, nvec, pitch, vec4);
}

// One matrix and one block of vectors, as a warp needs them.
struct BlockMat {
    const u32 *ptr, *row, *col, *lrow;
    const uint4 *chunk;
    const void *val;
    const uint4 *xs;    // rows of X, pitch words of 16 bytes each
    u64 *carry;
    u32 *count;
    u32 *y;
    long long ldy;
    int pitch, pieces, nvec, vec4, lgt;  // pieces of 16 bytes per row of X; lgt: log2 of the lanes that hold them
    u32 quad1;                    // rows r of the one-quad class: quad quad1 + r
    int fold;                     // m <= 2^31
    Mod M;
};

struct BlockArgs {
    BlockMat m;
    int nchunk_warps;             // warps 0 .. nchunk - 1 take the chunks
    u32 warp0[kBlockClasses + 1]; // first warp of each class, heaviest class first
    u32 row0[kBlockClasses + 1];  // its rows
    int lgg[kBlockClasses];       // log2 of groups per row
};

// Sums of one lane: 8 components of u16 residues (64-bit sums of terms below
// 2^32, at most 2^32 of them) or 4 of u32 residues (96-bit sums).
template <bool SMALL>
struct BlockAcc;

template <>
struct BlockAcc<true> {
    static constexpr int C = 8;
    typedef u64 Sum;
    u64 a[8];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = 0;
    }
    __device__ __forceinline__ void quad(const uint2 &vv, const uint4 (&x)[4], int)
    {
        const u32 v[4] = {vv.x & 0xffffu, vv.x >> 16, vv.y & 0xffffu, vv.y >> 16};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const u32 w[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[2 * i] += (u64)v[u] * (w[i] & 0xffffu);
                a[2 * i + 1] += (u64)v[u] * (w[i] >> 16);
            }
        }
    }
    static __device__ __forceinline__ u64 sel(bool b, u64 x, u64 y) { return b ? x : y; }
    static __device__ __forceinline__ u64 add_from(u64 keep, u64 send, int off)
    {
        return keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
    static __device__ __forceinline__ u32 get(u64 s, const Mod &M) { return red64(s, M); }
};

template <>
struct BlockAcc<false> {
    static constexpr int C = 4;
    typedef AccWide Sum;
    AccWide a[4];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i].zero();
    }
    __device__ __forceinline__ void quad(const uint4 &vv, const uint4 (&x)[4], int fold)
    {
        const u32 v[4] = {vv.x, vv.y, vv.z, vv.w};
        u32 w[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            w[u][0] = x[u].x;
            w[u][1] = x[u].y;
            w[u][2] = x[u].z;
            w[u][3] = x[u].w;
        }
        if (fold) {
            // m <= 2^31: four products, each below 2^62, in one 64-bit word
            // (a run-time test on purpose: it keeps the four gathers and the
            // next quad's loads ahead of the sums; as a template the sums
            // moved in between, 236 us against 191 at 16 vectors)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const u64 t = (u64)v[0] * w[0][i] + (u64)v[1] * w[1][i] + (u64)v[2] * w[2][i] + (u64)v[3] * w[3][i];
                asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, 0;"
                    : "+r"(a[i].w0), "+r"(a[i].w1), "+r"(a[i].w2)
                    : "r"((u32)t), "r"((u32)(t >> 32)));
            }
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i].mad(v[u], w[u][i]);
        }
    }
    static __device__ __forceinline__ AccWide sel(bool b, const AccWide &x, const AccWide &y)
    {
        AccWide r;
        r.w0 = b ? x.w0 : y.w0;
        r.w1 = b ? x.w1 : y.w1;
        r.w2 = b ? x.w2 : y.w2;
        return r;
    }
    static __device__ __forceinline__ AccWide add_from(AccWide keep, const AccWide &send, int off)
    {
        const u32 o0 = __shfl_xor_sync(0xffffffffu, send.w0, off), o1 = __shfl_xor_sync(0xffffffffu, send.w1, off),
                  o2 = __shfl_xor_sync(0xffffffffu, send.w2, off);
        asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
            : "+r"(keep.w0), "+r"(keep.w1), "+r"(keep.w2)
            : "r"(o0), "r"(o1), "r"(o2));
        return keep;
    }
    static __device__ __forceinline__ u32 get(const AccWide &s, const Mod &M) { return (u32)s.partial(M); }
};

// X is what the kernel before wrote, which may still run when this one starts
// (programmatic dependence): ordinary loads after the wait, never the read-only
// path, which is for data that nothing writes while the kernel runs.  COH: by
// way of L2 alone.
template <bool COH>
__device__ __forceinline__ uint4 block_gather(const char *p)
{
    if constexpr (COH) return __ldcg(reinterpret_cast<const uint4 *>(p));
    else return *reinterpret_cast<const uint4 *>(p);
}

// acc += quads k, k + step, ... below end; xb: this lane's piece of the rows
// of X.  Rows are padded to whole quads (value 0, column 0).
// X (and the y that earlier products read) belong to the kernel before this one
// in the stream: it is waited for with the first quad already on its way.
template <bool SMALL, bool COH>
__device__ __forceinline__ void block_entries(BlockAcc<SMALL> &acc, const BlockMat &a, u32 k, u32 end, u32 step,
                                              const char *xb, bool on)
{
    typedef typename std::conditional<SMALL, uint2, uint4>::type V;
    const u32 pb = (u32)a.pitch * 16u;
    uint4 j = make_uint4(0u, 0u, 0u, 0u);
    V v = V{};
    if (k < end) {
        j = __ldcs(reinterpret_cast<const uint4 *>(a.col) + k);
        v = __ldcs(reinterpret_cast<const V *>(a.val) + k);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if constexpr (COH) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next step may load its quads
    while (k < end) {
        uint4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = make_uint4(0u, 0u, 0u, 0u);
        if (on) {
            x[0] = block_gather<COH>(xb + (u64)j.x * pb);
            x[1] = block_gather<COH>(xb + (u64)j.y * pb);
            x[2] = block_gather<COH>(xb + (u64)j.z * pb);
            x[3] = block_gather<COH>(xb + (u64)j.w * pb);
        }
        // the next quad is on its way from memory while the gathers are
        const V vc = v;
        k += step;
        if (k < end) {
            j = __ldcs(reinterpret_cast<const uint4 *>(a.col) + k);
            v = __ldcs(reinterpret_cast<const V *>(a.val) + k);
        }
        acc.quad(vc, x, a.fold);
    }
}

// R consecutive components from column col0 of a row
template <int R>
__device__ __forceinline__ void block_write(const u32 (&r)[R], const BlockMat &a, u32 row, int col0)
{
    u32 *yp = a.y + (long long)row * a.ldy + col0;
    if (R >= 4 && a.vec4 && col0 + R <= a.nvec) {
#pragma unroll
        for (int i = 0; i + 4 <= R; i += 4) {
            u32 o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = combine(r[i + k], yp + i + k, false, a.M);
            __stcs(reinterpret_cast<uint4 *>(yp + i), make_uint4(o[0], o[1], o[2], o[3]));
        }
    } else {
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (col0 + i < a.nvec) yp[i] = combine(r[i], yp + i, false, a.M);
    }
}

// The sums of the 2^lgg groups of a row (lanes a multiple of T apart), each
// component in one group only: every step sends one half of the components
// to the partner and keeps the other.  R components, from `col0` on, are left
// in s when the steps S .. end; `emit(s, col0)` takes them from the lanes
// that hold final sums.
template <bool SMALL, int R, class Emit>
__device__ __forceinline__ void block_reduce(typename BlockAcc<SMALL>::Sum (&s)[R], int lgt, int lgg, int step, int lane,
                                             int col0, Emit emit)
{
    typedef BlockAcc<SMALL> A;
    if (step == lgg) {
        u32 o[R];
#pragma unroll
        for (int i = 0; i < R; ++i) o[i] = A::get(s[i], *emit.M);
        emit(o, col0);
        return;
    }
    const int off = 1 << (lgt + step);
    if constexpr (R > 1) {
        const bool up = (lane & off) != 0;
        typename A::Sum t[R / 2];
#pragma unroll
        for (int i = 0; i < R / 2; ++i)
            t[i] = A::add_from(A::sel(up, s[i + R / 2], s[i]), A::sel(up, s[i], s[i + R / 2]), off);
        block_reduce<SMALL, R / 2>(t, lgt, lgg, step + 1, lane, col0 + (up ? R / 2 : 0), emit);
    } else {
        // one component left: the lanes of the remaining steps all get the sum
        for (; step < lgg; ++step) s[0] = A::add_from(s[0], s[0], 1 << (lgt + step));
        // ... and the one whose bits of those steps are 0 writes it
        constexpr int full = SMALL ? 3 : 2;
        const bool mine = (lane & (((1 << lgg) - (1 << full)) << lgt)) == 0;
        u32 o[1] = {A::get(s[0], *emit.M)};
        if (mine) emit(o, col0);
    }
}

struct BlockEmitRow {
    const BlockMat *a;
    const Mod *M;
    u32 row;
    bool ok;
    template <int R>
    __device__ __forceinline__ void operator()(const u32 (&o)[R], int col0) const
    {
        if (ok) block_write<R>(o, *a, row, col0);
    }
};

struct BlockEmitCarry {
    const BlockMat *a;
    const Mod *M;
    u64 *cw;
    template <int R>
    __device__ __forceinline__ void operator()(const u32 (&o)[R], int col0) const
    {
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (col0 + i < a->nvec) atomicAdd(cw + col0 + i, (u64)o[i]);
    }
};

// A warp's chunk of a long row.
template <bool SMALL, bool COH = false>
__device__ __forceinline__ void block_chunk(const BlockMat &a, u32 w, int lane)
{
    constexpr int C = BlockAcc<SMALL>::C;
    const int T = 1 << a.lgt, c = lane & (T - 1);
    BlockAcc<SMALL> acc;
    acc.zero();
    const uint4 ch = __ldg(a.chunk + w);
    block_entries<SMALL, COH>(acc, a, ch.y + (u32)(lane >> a.lgt), ch.z, 32u >> a.lgt,
                         reinterpret_cast<const char *>(a.xs + c), c < a.pieces);
    u64 *cw = a.carry + (size_t)ch.x * kBlockVecs;
    const BlockEmitCarry emit = {&a, &a.M, cw};
    block_reduce<SMALL, C>(acc.a, a.lgt, 5 - a.lgt, 0, lane, c * C, emit);
    // the chunk that arrives last writes the row and clears its words
    u32 last = 0;
    __threadfence();
    __syncwarp();
    u32 *count = a.count + (size_t)ch.x * kBlockVecs;
    if (lane == 0) last = atomicAdd(count, 1u) == ch.w - 1u ? 1u : 0u;
    last = __shfl_sync(0xffffffffu, last, 0);
    if (!last) return;
    __threadfence();
    const u32 row = __ldg(a.lrow + ch.x);
    if (lane < a.nvec) {
        u32 *yp = a.y + (long long)row * a.ldy + lane;
        *yp = combine(red64(__ldcg(cw + lane), a.M), yp, false, a.M);
        cw[lane] = 0;
    }
    if (lane == 0) *count = 0;
}

// A warp's 32 / (T G) rows of a class: r0 the first, below rend, G = 2^lgg.
template <bool SMALL, bool COH = false>
__device__ __forceinline__ void block_rows(const BlockMat &a, u32 r0, u32 rend, int lgg, bool one, int lane)
{
    constexpr int C = BlockAcc<SMALL>::C;
    const int T = 1 << a.lgt, c = lane & (T - 1), lgr = a.lgt + lgg;
    const bool on = c < a.pieces;
    BlockAcc<SMALL> acc;
    acc.zero();
    const u32 r = r0 + (u32)(lane >> lgr);
    BlockEmitRow emit = {&a, &a.M, 0u, r < rend && on};
    u32 s = 0, e = 0;
    if (r < rend) {
        // rows of one quad lie one after another: no offset to wait for
        s = one ? a.quad1 + r : __ldg(a.ptr + r);
        e = one ? s + 1u : __ldg(a.ptr + r + 1);
        emit.row = __ldg(a.row + r);
    }
    block_entries<SMALL, COH>(acc, a, s + (u32)((lane >> a.lgt) & ((1 << lgg) - 1)), e, 1u << lgg,
                              reinterpret_cast<const char *>(a.xs + c), on);
    block_reduce<SMALL, C>(acc.a, a.lgt, lgg, 0, lane, c * C, emit);
}

// The rows of warp w >= nchunk_warps.
template <bool SMALL, bool COH>
__device__ __forceinline__ void block_class_rows(const BlockArgs &a, u32 w, int lane)
{
    // the class of this warp (warp0 grows; the last entry ends the list)
    int b = 0;
#pragma unroll
    for (int i = 1; i < kBlockClasses; ++i)
        if (w >= a.warp0[i]) b = i;
    if (w >= a.warp0[kBlockClasses]) return;
    const int lgg = a.lgg[b];
    block_rows<SMALL, COH>(a.m, a.row0[b] + ((w - a.warp0[b]) << (5 - a.m.lgt - lgg)), a.row0[b + 1], lgg,
                           b == kBlockClasses - 2, lane);
}

template <bool SMALL>
__global__ void __launch_bounds__(kBlockThreads, 4) k_block(const __grid_constant__ BlockArgs a)
{
    const u32 w = blockIdx.x * (kBlockThreads / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (w < (u32)a.nchunk_warps) {
        block_chunk<SMALL>(a.m, w, lane);
        return;
    }
    block_class_rows<SMALL, false>(a, w, lane);
}

// One step of a block sequence at m > 2^16: V_{i+1} = A V_i and S_i = X^T V_i in
// one launch, both read V_i.  CTAs below `spmm` multiply; each of the next
// `proj` projects its rows (four outputs of one row of S per thread, the
// threads in groups that take every ngrp-th row) and writes its reduced sums;
// the last `fin` add up the sums of the step before, kStepOuts outputs each, and
// write S_{i-1}, so that no CTA waits for another (one CTA for all 1 024 outputs
// of s = 32 was the longest of the launch: 59 us per step at 4 001 rows).  V: rows of ldv words (a multiple of four, zero past
// s).  A kernel lets the next one start once the one before it is complete.
constexpr int kStepOuts = 64;
struct BlockStep {
    BlockArgs b;
    unsigned spmm, proj, fin; // CTAs of each kind
    int s, tiles, ngrp;       // tiles of four outputs, groups of threads
    long long n, ldv, per;    // rows, words per row of V, rows per projecting CTA
    const u32 *X, *V;
    u32 *part, *prev;         // [proj][s s]: this step's sums, the step before's (null: none)
    u32 *S;                   // S_{i-1}
};

__global__ void __launch_bounds__(kBlockThreads, 3) k_block_step(const __grid_constant__ BlockStep a)
{
    __shared__ __align__(8) u32 red[4 * kBlockThreads];
    const int tid = threadIdx.x;
    if (blockIdx.x < a.spmm) {
        const u32 w = blockIdx.x * (kBlockThreads / 32) + (tid >> 5);
        if (w < (u32)a.b.nchunk_warps) block_chunk<false, true>(a.b.m, w, tid & 31);
        else if (w < a.b.warp0[kBlockClasses]) block_class_rows<false, true>(a.b, w, tid & 31);
        return;
    }
    const Mod &M = a.b.m.M;
    const int outs = a.s * a.s;
    if (blockIdx.x >= gridDim.x - a.fin) {
        // an output's sums by kBlockThreads / kStepOuts threads
        constexpr int kParts = kBlockThreads / kStepOuts;
        const int o = (int)(blockIdx.x - (gridDim.x - a.fin)) * kStepOuts + tid % kStepOuts;
        u64 *part = reinterpret_cast<u64 *>(red), sum = 0;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (!a.prev) return;
        if (o < outs) {
#pragma unroll 8
            for (unsigned c = tid / kStepOuts; c < a.proj; c += kParts) sum += __ldcg(a.prev + (size_t)c * outs + o);
        }
        part[tid] = sum;
        __syncthreads();
        if (tid < kStepOuts && o < outs) {
#pragma unroll
            for (int k = 1; k < kParts; ++k) sum += part[k * kStepOuts + tid];
            a.S[o] = red64(sum, M);
        }
        return;
    }
    const long long r0 = (long long)(blockIdx.x - a.spmm) * a.per, r1 = min(a.n, r0 + a.per);
    const int g = tid / a.tiles, t = tid - g * a.tiles, bt = (a.s + 3) / 4;   // tile: row t / bt of S, columns 4 (t mod bt) ..
    const int ai = t / bt, c0 = 4 * (t - ai * bt);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    AccWide acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i].zero();
    if (g < a.ngrp) {
#pragma unroll 4
        for (long long r = r0 + g; r < r1; r += a.ngrp) {
            const u32 x = __ldg(a.X + r * a.s + ai);
            const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(a.V + r * a.ldv + c0));
            acc[0].mad(x, v.x);
            acc[1].mad(x, v.y);
            acc[2].mad(x, v.z);
            acc[3].mad(x, v.w);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) red[i * kBlockThreads + tid] = g < a.ngrp ? (u32)acc[i].partial(M) : 0u;
    __syncthreads();
    if (tid < a.tiles) {
        u32 *dst = a.part + (size_t)(blockIdx.x - a.spmm) * outs + ai * a.s;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            u64 sum = 0;
            for (int k = 0; k < a.ngrp; ++k) sum += red[i * kBlockThreads + k * a.tiles + tid];
            if (c0 + i < a.s) dst[c0 + i] = red64(sum, M);
        }
    }
}

// Many matrices in one launch, each with its modulus, vectors and packed X:
// what a launch passes for one of them, and the first warp (or, for the
// staging, the first CTA) of each.
constexpr int kMany = 512;
struct BlockMany {
    const BlockDev *dev[kMany];
    const u32 *x[kMany];
    uint4 *xs[kMany];
    u32 *y[kMany];
    u32 first[kMany + 1];
    unsigned char nvec[kMany];                // bit 7: x is read where it lies, else packed in xs
    unsigned char v0[kMany];                  // first word of each long row's sums (a matrix that is there twice)
    int count;
};
static_assert(sizeof(BlockMany) < 32000, "launch parameters");

__device__ __forceinline__ int block_find(const BlockMany &P, u32 w)
{
    int lo = 0, hi = P.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.first[mid] <= w) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(kBlockThreads) k_block_stage_many(const __grid_constant__ BlockMany P)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int j = block_find(P, blockIdx.x);
    const BlockDev &D = *P.dev[j];
    const int nvec = P.nvec[j], C = D.small ? 8 : 4, pieces = (nvec + C - 1) / C;
    const u32 *x = P.x[j];
    const int vec4 = nvec % 4 == 0 && ((uintptr_t)x & 15u) == 0;
    const long long t = (long long)(blockIdx.x - P.first[j]) * kBlockThreads + threadIdx.x;
    if (t >= D.ncols * pieces) return;
    P.xs[j][t] = D.small ? block_pack<true>(x, nvec, t, nvec, pieces, vec4) : block_pack<false>(x, nvec, t, nvec, pieces, vec4);
}

__global__ void __launch_bounds__(kBlockThreads, 4) k_block_many(const __grid_constant__ BlockMany P)
{
    const u32 w0 = blockIdx.x * (kBlockThreads / 32) + (threadIdx.x >> 5);
    if (w0 >= P.first[P.count]) return;
    const int lane = threadIdx.x & 31, j = block_find(P, w0);
    const BlockDev &D = *P.dev[j];
    BlockMat a;
    a.ptr = D.ptr;
    a.row = D.row;
    a.col = D.col;
    a.lrow = D.lrow;
    a.chunk = D.chunk;
    a.val = D.val;
    a.carry = D.carry + P.v0[j];
    a.count = D.count + P.v0[j];
    a.y = P.y[j];
    a.nvec = P.nvec[j] & 127;
    a.ldy = a.nvec;
    const int C = D.small ? 8 : 4;
    a.pieces = (a.nvec + C - 1) / C;
    a.lgt = a.pieces > 1 ? 32 - __clz(a.pieces - 1) : 0;
    a.xs = P.nvec[j] & 128 ? reinterpret_cast<const uint4 *>(P.x[j]) : P.xs[j];
    a.pitch = a.pieces;
    a.vec4 = a.nvec % 4 == 0 && ((uintptr_t)a.y & 15u) == 0;
    a.quad1 = D.quad1;
    a.fold = D.fold;
    a.M = D.M;
    u32 w = w0 - P.first[j];
    if (w < D.nchunk) {
        if (D.small) block_chunk<true>(a, w, lane);
        else block_chunk<false>(a, w, lane);
        return;
    }
    w -= D.nchunk;
    int b = 0, lgg = 0;
    u32 r0 = 0, rend = 0;
    for (; b < kBlockClasses; ++b) {
        r0 = D.row0[b];
        rend = D.row0[b + 1];
        lgg = block_lgg(b, a.lgt);
        const int sh = 5 - a.lgt - lgg;
        const u32 nw = (u32)(((u64)(rend - r0) + (1u << sh) - 1u) >> sh);
        if (w < nw) {
            r0 += w << sh;
            break;
        }
        w -= nw;
    }
    if (b == kBlockClasses) return;
    if (D.small) block_rows<true>(a, r0, rend, lgg, b == kBlockClasses - 2, lane);
    else block_rows<false>(a, r0, rend, lgg, b == kBlockClasses - 2, lane);
}

// x is read in place where its rows already are whole aligned 16-byte pieces of
// u32, else packed by a launch before.
bool block_in_place(bool small, const u32 *x, long long ldx, int nv)
{
    return !small && nv % 4 == 0 && ldx % 4 == 0 && ((uintptr_t)x & 15u) == 0 && ldx / 4 < (1LL << 28);
}

// log2 of the 16-byte pieces per packed row that a block's widest packed pass
// takes, rounded up; -1 when all of it is read in place
int staging_width(bool small, const u32 *x, long long ldx, int nvec)
{
    const int C = small ? 8 : 4, last = (nvec - 1) % kBlockVecs + 1;   // vectors of the last pass
    int pieces = 0, lg = -1;
    if (nvec > kBlockVecs && !block_in_place(small, x, ldx, kBlockVecs)) pieces = kBlockVecs / C;
    else if (!block_in_place(small, x + (nvec - last), ldx, last)) pieces = (last + C - 1) / C;
    for (; pieces; pieces = pieces > 1 ? (pieces + 1) / 2 : 0) ++lg;
    return lg;
}

// ---------------------------------------------------------------------------
// Layouts are made on the device from the CSR arrays, any number at a time (a
// job each, blockIdx.y): the lengths of the output rows (of A: row offsets; of
// A^T: a histogram of the columns), the rows and quads of each class, each
// row's place (a warp's rows of a class take consecutive places, so rows stay
// nearly in order) with its padding, then the entries.  The order of the
// entries of a row is free: sums mod m are exact.
struct BlockBuild {
    const long long *ptr;   // CSR of A
    const u32 *col, *val;   // val null: all odd
    long long nr, n;        // rows of A, output rows
    u32 *len, *start;       // [n]: entries, first quad
    u64 *cursor;            // [kBlockClasses + 2]: (rows << 32) + quads of each class and of the long rows; chunks
    u32 *orow, *optr, *lrow, *ocol;
    uint4 *chunk;
    void *oval;
    int small, odd, transpose;   // odd: the pattern of the odd values only, without values
    u32 rows, quads;        // of the layout, without and with the long rows
    BlockDev dev, *dev_out;
};

__global__ void __launch_bounds__(kBlockThreads) k_block_lengths(const BlockBuild *__restrict__ jobs)
{
    const BlockBuild &b = jobs[blockIdx.y];
    const long long nth = (long long)gridDim.x * kBlockThreads, t = (long long)blockIdx.x * kBlockThreads + threadIdx.x;
    const bool odd = b.odd && b.val;   // some of the values do not count
    if (!b.transpose && !odd) {
        for (long long i = t; i < b.nr; i += nth) b.len[i] = (u32)(b.ptr[i + 1] - b.ptr[i]);
    } else if (!b.transpose) {
        for (long long w = t >> 5; w < b.nr; w += nth >> 5) {   // a warp per row
            const long long e = b.ptr[w + 1];
            u32 c = 0;
            for (long long k = b.ptr[w] + (threadIdx.x & 31); k < e; k += 32) c += b.val[k] & 1u;
            c = __reduce_add_sync(0xffffffffu, c);
            if ((threadIdx.x & 31) == 0) b.len[w] = c;
        }
    } else {
        const long long nnz = b.ptr[b.nr];
        for (long long k = t; k < nnz; k += nth)
            if (!odd || (b.val[k] & 1u)) atomicAdd(b.len + b.col[k], 1u);
    }
}

// place = 0: the totals of every class into the cursors; place = 1: every row
// to its place, the cursors holding the first places.
__global__ void __launch_bounds__(kBlockThreads) k_block_place(const BlockBuild *__restrict__ jobs, int place)
{
    const BlockBuild &b = jobs[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const long long n = b.n, nw = (n + 31) / 32, step = (long long)gridDim.x * (kBlockThreads / 32);
    for (long long w = (long long)blockIdx.x * (kBlockThreads / 32) + (threadIdx.x >> 5); w < nw; w += step) {
        const long long i = w * 32 + lane;
        const u32 len = i < n ? b.len[i] : 0u, quads = (u32)(((u64)len + 3u) / 4u);
        const int c = i >= n ? -1 : len > (u32)kBlockLong ? kBlockClasses : block_class(quads);
        const u32 parts = c == kBlockClasses ? (u32)(((u64)len + kBlockLong - 1) / kBlockLong) : 0u;
        for (int k = 0; k <= kBlockClasses; ++k) {
            const u32 same = __ballot_sync(0xffffffffu, c == k);
            if (!same) continue;
            // this lane's offset among the warp's rows of the class
            u64 mine = c == k ? ((u64)1 << 32) + quads : 0, sum = mine;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const u64 o = __shfl_up_sync(0xffffffffu, sum, d);
                if (lane >= d) sum += o;
            }
            const u64 all = __shfl_sync(0xffffffffu, sum, 31);
            u64 base = 0;
            if (lane == 0) base = atomicAdd(b.cursor + k, all);
            base = __shfl_sync(0xffffffffu, base, 0);
            if (c != k) continue;
            if (!place) {
                if (parts) atomicAdd(b.cursor + kBlockClasses + 1, (u64)parts);
                continue;
            }
            const u64 at = base + sum - mine;
            const u32 slot = (u32)(at >> 32), q = (u32)at;
            b.start[i] = q;
            // padding entries (value 0, or no column)
            for (size_t e = (size_t)q * 4 + len, end = ((size_t)q + quads) * 4; e < end; ++e) {
                b.ocol[e] = b.odd ? 0xffffffffu : 0u;
                if (b.odd) continue;
                if (b.small) reinterpret_cast<unsigned short *>(b.oval)[e] = 0;
                else reinterpret_cast<u32 *>(b.oval)[e] = 0u;
            }
            if (k == kBlockClasses) {
                b.lrow[slot] = (u32)i;
                for (int v = 0; v < kBlockVecs && !b.odd; ++v) {
                    b.dev.carry[(size_t)slot * kBlockVecs + v] = 0;
                    b.dev.count[(size_t)slot * kBlockVecs + v] = 0u;
                }
                const u64 c0 = atomicAdd(b.cursor + kBlockClasses + 1, (u64)parts);
                for (u32 p = 0; p < parts; ++p)
                    b.chunk[c0 + p] = make_uint4(slot, q + p * (u32)(kBlockLong / 4),
                                                 q + min(quads, (p + 1) * (u32)(kBlockLong / 4)), parts);
            } else {
                b.orow[slot] = (u32)i;
                b.optr[slot] = q;
            }
        }
    }
}

__global__ void __launch_bounds__(kBlockThreads) k_block_fill(const BlockBuild *__restrict__ jobs)
{
    const BlockBuild &b = jobs[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const bool transpose = b.transpose != 0, small = b.small != 0, values = b.odd == 0, odd = !values && b.val;
    if (blockIdx.x == 0 && threadIdx.x == 0 && b.dev_out) {
        *b.dev_out = b.dev;
        b.optr[b.rows] = b.quads;
    }
    const long long step = (long long)gridDim.x * (kBlockThreads / 32);
    for (long long i = (long long)blockIdx.x * (kBlockThreads / 32) + (threadIdx.x >> 5); i < b.nr; i += step) {
        const long long s = b.ptr[i], e = b.ptr[i + 1];
        for (long long k = s + lane; k < e; k += 32) {
            const u32 j = b.col[k], v = values || odd ? b.val[k] : 1u;
            if (odd && !(v & 1u)) continue;
            const u32 r = transpose ? j : (u32)i;
            const size_t to = (size_t)b.start[r] * 4 +
                              (transpose || odd ? (size_t)(atomicSub(b.len + r, 1u) - 1u) : (size_t)(k - s));
            b.ocol[to] = transpose ? (u32)i : j;
            if (!values) continue;
            if (small) reinterpret_cast<unsigned short *>(b.oval)[to] = (unsigned short)v;
            else reinterpret_cast<u32 *>(b.oval)[to] = v;
        }
    }
}

bool capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) return false;
    cudaGetLastError();
    return true;
}

// A layout to be made: of A (nr x nc, values below m), or of A^T, with a buffer
// for packed rows of 2^lgx pieces (lgx = -1: none).
struct BlockJob {
    BlockPlan *B;
    const ffspmv_handle *h;
    bool transpose, odd;
    int lgx;
    ffspmv_status st;
};

ffspmv_status block_limits(const BlockJob &J)
{
    const long long nr = J.h->A.nrows, *ptr = J.h->h_ptr.data(), nnz = ptr[nr], n = J.transpose ? J.h->A.ncols : nr;
    const int *col = J.h->h_col.data();
    // offsets in quads and lengths of rows are 32-bit; with values, 32-bit row numbers are rounded up to a warp's
    constexpr long long kLim = (1LL << 32) - 1;
    if (nnz / 4 + std::min(n, nnz) >= kLim || (!J.odd && (nnz >= kLim || n >= kLim - 63))) return FFSPMV_ERR_UNSUPPORTED;
    if (nnz >= kLim) {
        std::vector<long long> len((size_t)n, 0);
        for (long long i = 0; i < nr; ++i)
            for (long long k = ptr[i]; k < ptr[i + 1]; ++k) ++len[J.transpose ? (size_t)col[k] : (size_t)i];
        for (long long l : len)
            if (l >= kLim) return FFSPMV_ERR_UNSUPPORTED;
    }
    return FFSPMV_OK;
}

// Uploads of a handle's arrays go through page-locked memory.  The copy engine
// reads pageable memory at 130 GB/s on a good day, but it makes the pages it
// touches candidates for migration, and once that has begun the 126 MB of a
// 15.8M-entry matrix take 20 to 45 ms.  Here kUpLanes host threads fill a slot
// each and send it (one thread copies 12 to 16 GB/s, four 55): 5.3 ms for the
// whole first block.  Builds of less than kUpLeast bytes do without: locking the
// buffer and starting the threads takes 0.5 ms (2.7M entries: 0.8 ms without on a
// good day, 1.3 with).
constexpr int kUpLanes = 4;
constexpr size_t kUpSlot = 1 << 20, kUpDirect = 64 * 1024;   // smaller copies leave the host's memory at once
constexpr size_t kUpLeast = 32 << 20;

// What the library keeps while it has handles: that buffer, used by one build at
// a time, and per device a pool for the builds' temporary memory (up to
// kKeepPool bytes of it: a default pool gives all of it back at once, 0.2 ms).
constexpr int kKeepDevices = 16;
constexpr unsigned long long kKeepPool = 32ull << 20;
struct BlockKeep {
    std::mutex use;      // of buf
    std::mutex state;    // of the rest
    long long handles = 0;
    char *buf = nullptr;
    cudaMemPool_t pool[kKeepDevices] = {};
};
BlockKeep &block_keep()
{
    static BlockKeep *k = new BlockKeep();   // (outlives the handles of a process that ends without freeing them)
    return *k;
}

// The current device's pool; null: the default one.
cudaMemPool_t block_pool()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kKeepDevices) return nullptr;
    BlockKeep &K = block_keep();
    std::lock_guard<std::mutex> lock(K.state);
    if (!K.pool[dev]) {
        cudaMemPoolProps p = {};
        p.allocType = cudaMemAllocationTypePinned;
        p.location.type = cudaMemLocationTypeDevice;
        p.location.id = dev;
        unsigned long long keep = kKeepPool;
        if (cudaMemPoolCreate(&K.pool[dev], &p) != cudaSuccess) {
            cudaGetLastError();
            K.pool[dev] = nullptr;
        } else {
            cudaMemPoolSetAttribute(K.pool[dev], cudaMemPoolAttrReleaseThreshold, &keep);
        }
    }
    return K.pool[dev];
}

class BlockUpload {
    struct Piece {
        char *dst;
        const char *src;
        size_t bytes;
    };
    std::unique_lock<std::mutex> lock;
    std::vector<Piece> pieces;   // at most kUpSlot bytes each
    cudaStream_t st;
    cudaEvent_t sent[kUpLanes] = {};
    char *buf = nullptr;

    // pieces k, k + kUpLanes, ... through slot k
    cudaError_t lane(int k) const
    {
        char *h = buf + (size_t)k * kUpSlot;
        for (size_t i = (size_t)k; i < pieces.size(); i += kUpLanes) {
            const Piece &p = pieces[i];
            cudaError_t e = cudaEventSynchronize(sent[k]);   // (never recorded: done)
            if (e != cudaSuccess) return e;
            memcpy(h, p.src, p.bytes);
            if ((e = cudaMemcpyAsync(p.dst, h, p.bytes, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
            if ((e = cudaEventRecord(sent[k], st)) != cudaSuccess) return e;
        }
        return cudaSuccess;
    }

public:
    BlockUpload(cudaStream_t s, size_t bytes) : st(s)
    {
        if (bytes < kUpLeast) return;
        pieces.reserve(bytes / kUpSlot + 64);
        BlockKeep &K = block_keep();
        lock = std::unique_lock<std::mutex>(K.use);
        if (!K.buf && cudaHostAlloc((void **)&K.buf, kUpLanes * kUpSlot, cudaHostAllocPortable) != cudaSuccess) K.buf = nullptr;
        bool ok = K.buf != nullptr;
        for (cudaEvent_t &e : sent) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
        if (ok) buf = K.buf;
        cudaGetLastError();   // (without it: ordinary copies)
    }
    ~BlockUpload()
    {
        cudaStreamSynchronize(st);   // the next build may fill the slots, the sources may go
        for (cudaEvent_t e : sent)
            if (e) cudaEventDestroy(e);
    }
    BlockUpload(const BlockUpload &) = delete;

    // The copy is made by send() unless it is small.
    ffspmv_status copy(void *dst, const void *src, size_t bytes)
    {
        if (!bytes) return FFSPMV_OK;
        if (!buf || bytes < kUpDirect) {
            FF_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st));
            return FFSPMV_OK;
        }
        for (size_t at = 0; at < bytes; at += kUpSlot)
            pieces.push_back({(char *)dst + at, (const char *)src + at, std::min(kUpSlot, bytes - at)});
        return FFSPMV_OK;
    }
    ffspmv_status send()
    {
        cudaError_t err[kUpLanes] = {};
        std::thread helper[kUpLanes];
        int dev = 0;
        cudaGetDevice(&dev);
        // a thread is worth starting for a few pieces
        const int helpers = pieces.size() >= 4 * kUpLanes ? kUpLanes - 1 : 0;
        for (int k = 0; k < helpers; ++k)
            try {
                helper[k] = std::thread([this, k, dev, &err] {
                    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
                    cudaThreadExchangeStreamCaptureMode(&mode);
                    if ((err[k] = cudaSetDevice(dev)) == cudaSuccess) err[k] = lane(k);
                });
            } catch (const std::exception &) {   // no thread: this one does it
            }
        for (int k = kUpLanes - 1; k >= 0; --k) {
            if (helper[k].joinable()) helper[k].join();
            else err[k] = lane(k);
        }
        for (cudaError_t e : err) FF_CUDA(e);
        return FFSPMV_OK;
    }
};

// What a build holds: a stream of its own, so that nothing waits for the
// caller's, temporary memory in that stream's order (a cudaFree would wait for
// all of them), and this thread's leave to allocate while another stream is
// being captured.
struct BlockScope {
    cudaStream_t st = nullptr;
    void *tmp = nullptr;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    BlockScope() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~BlockScope()
    {
        if (tmp) cudaFreeAsync(tmp, st);
        if (st) {
            cudaStreamSynchronize(st);
            cudaStreamDestroy(st);
        }
        cudaThreadExchangeStreamCaptureMode(&mode);
    }
};

constexpr int kBlockCursors = kBlockClasses + 2;
constexpr size_t kBlockAlign = 256;
size_t block_round(size_t b) { return (std::max<size_t>(b, 16) + kBlockAlign - 1) / kBlockAlign * kBlockAlign; }

// Device memory that a job's arrays take while it is built.
size_t block_job_bytes(const BlockJob &J)
{
    const size_t nr = (size_t)J.h->A.nrows, n = J.transpose ? (size_t)J.h->A.ncols : nr, nnz = J.h->h_col.size();
    return block_round((nr + 1) * 8) + 2 * block_round(nnz * 4) + 2 * block_round(n * 4);
}

// The layouts of all the jobs (within the limits), with two synchronisations of
// the build's stream in all.  Arrays below kPack bytes go up together.
ffspmv_status build_blocks(BlockJob *jobs, int count, BlockScope &S)
{
    constexpr size_t kPack = 256 * 1024;
    FF_CUDA(cudaStreamCreateWithFlags(&S.st, cudaStreamNonBlocking));
    cudaStream_t st = S.st;
    std::vector<BlockBuild> b((size_t)count);
    memset(b.data(), 0, sizeof(BlockBuild) * b.size());
    // [jobs][cursors][small arrays] (one copy), [large arrays], [lengths], [first quads]
    const size_t o_cur = block_round(sizeof(BlockBuild) * b.size()),
                 head = o_cur + block_round(sizeof(u64) * kBlockCursors * b.size());
    struct Array {
        const void *src;
        size_t bytes, at;
    };
    std::vector<Array> arr((size_t)3 * count);
    for (int j = 0; j < count; ++j) {
        const ffspmv_handle &h = *jobs[j].h;
        arr[3 * j] = {h.h_ptr.data(), h.h_ptr.size() * 8, 0};
        arr[3 * j + 1] = {h.h_col.data(), h.h_col.size() * 4, 0};
        // (a pattern of odd values needs none of them when all are)
        arr[3 * j + 2] = {h.h_val.data(), jobs[j].odd && h.all_odd ? 0 : h.h_val.size() * 4, 0};
    }
    size_t o = head;
    for (Array &a : arr)
        if (a.bytes < kPack) {
            a.at = o;
            o += block_round(a.bytes);
        }
    const size_t packed = o;
    for (Array &a : arr)
        if (a.bytes >= kPack) {
            a.at = o;
            o += block_round(a.bytes);
        }
    const size_t o_len = o;
    long long most = 1;
    std::vector<size_t> lens((size_t)count), starts((size_t)count);
    for (int pass = 0; pass < 2; ++pass)
        for (int j = 0; j < count; ++j) {
            const long long n = jobs[j].transpose ? jobs[j].h->A.ncols : jobs[j].h->A.nrows;
            (pass ? starts : lens)[j] = o;
            o += block_round((size_t)n * 4);
            most = std::max(most, std::max(n, jobs[j].h->A.nrows));
        }
    const size_t o_start = starts[0];
    const cudaMemPool_t pool = block_pool();
    if ((pool ? cudaMallocFromPoolAsync(&S.tmp, o, pool, st) : cudaMallocAsync(&S.tmp, o, st)) != cudaSuccess) {
        cudaGetLastError();
        S.tmp = nullptr;
        return FFSPMV_ERR_OOM;
    }
    char *t = (char *)S.tmp;
    for (int j = 0; j < count; ++j) {
        const BlockJob &J = jobs[j];
        b[j].ptr = (const long long *)(t + arr[3 * j].at);
        b[j].col = (const u32 *)(t + arr[3 * j + 1].at);
        b[j].val = arr[3 * j + 2].bytes ? (const u32 *)(t + arr[3 * j + 2].at) : nullptr;
        b[j].nr = J.h->A.nrows;
        b[j].n = J.transpose ? J.h->A.ncols : J.h->A.nrows;
        b[j].len = (u32 *)(t + lens[j]);
        b[j].start = (u32 *)(t + starts[j]);
        b[j].cursor = (u64 *)(t + o_cur) + (size_t)j * kBlockCursors;
        b[j].small = J.h->m <= 65536u ? 1 : 0;
        b[j].odd = J.odd ? 1 : 0;
        b[j].transpose = J.transpose ? 1 : 0;
    }
    // host ends of copies, here so that none is freed while one goes on
    // (to_device waits for the stream when it goes)
    std::vector<char> up(packed, 0);
    std::vector<u64> curs((size_t)kBlockCursors * count);
    memcpy(up.data(), b.data(), sizeof(BlockBuild) * b.size());
    for (const Array &a : arr)
        if (a.bytes && a.bytes < kPack) memcpy(up.data() + a.at, a.src, a.bytes);
    BlockUpload to_device(st, o);
    ffspmv_status r = to_device.copy(t, up.data(), packed);
    for (const Array &a : arr)
        if (r == FFSPMV_OK && a.bytes >= kPack) r = to_device.copy(t + a.at, a.src, a.bytes);
    if (r == FFSPMV_OK) r = to_device.send();
    if (r != FFSPMV_OK) return r;
    FF_CUDA(cudaMemsetAsync(t + o_len, 0, o_start - o_len, st));
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const dim3 grid((unsigned)std::min<long long>(8 * std::max(nsm, 1), (most + 7) / 8), (unsigned)count);
    const BlockBuild *dj = (const BlockBuild *)t;
    k_block_lengths<<<grid, kBlockThreads, 0, st>>>(dj);
    k_block_place<<<grid, kBlockThreads, 0, st>>>(dj, 0);
    FF_CUDA(cudaGetLastError());
    FF_CUDA(cudaMemcpyAsync(curs.data(), t + o_cur, sizeof(u64) * curs.size(), cudaMemcpyDeviceToHost, st));
    FF_CUDA(cudaStreamSynchronize(st));
    for (int j = 0; j < count; ++j) {
        BlockJob &J = jobs[j];
        BlockPlan &B = *J.B;
        u64 *cur = curs.data() + (size_t)j * kBlockCursors;
        const u32 m = J.h->m;
        // the long rows' quads come first, then the classes, heaviest first
        B.n = b[j].n;
        B.ncols = J.transpose ? J.h->A.nrows : J.h->A.ncols;
        B.small = b[j].small != 0;
        B.nsm = std::max(nsm, 1);
        B.nlong = (long long)(cur[kBlockClasses] >> 32);
        B.nchunk = (long long)cur[kBlockClasses + 1];
        u64 quads = cur[kBlockClasses] & 0xffffffffull, rows = 0;
        cur[kBlockClasses] = cur[kBlockClasses + 1] = 0;
        for (int i = 0; i < kBlockClasses; ++i) {
            const int c = kBlockClasses - 1 - i;
            const u64 here = cur[c];
            cur[c] = (rows << 32) + quads;
            if (c == 1) B.quad1 = (u32)quads - (u32)rows;
            rows += here >> 32;
            quads += here & 0xffffffffull;
            B.cls_row[i + 1] = (long long)rows;
        }
        const int vb = J.odd ? 0 : B.small ? 2 : 4;
        size_t a = 0;
        auto put = [&](size_t bytes) {
            const size_t here = a;
            a += block_round(bytes);
            return here;
        };
        const size_t o_ptr = put((size_t)(rows + 1) * 4), o_row = put((size_t)rows * 4), o_chunk = put((size_t)B.nchunk * 16),
                     o_lrow = put((size_t)B.nlong * 4), o_col = put((size_t)quads * 16), o_val = put((size_t)quads * 4 * vb),
                     o_carry = put((size_t)(J.odd ? 0 : B.nlong) * kBlockVecs * 8),
                     o_count = put((size_t)(J.odd ? 0 : B.nlong) * kBlockVecs * 4),
                     o_dev = put(sizeof(BlockDev)),
                     o_xs = put(J.lgx < 0 ? 0 : ((size_t)B.ncols << J.lgx) * sizeof(uint4));
        if (cudaMalloc(&B.arena, a) != cudaSuccess) {
            cudaGetLastError();
            B.arena = nullptr;
            J.st = FFSPMV_ERR_OOM;
            b[j].nr = b[j].n = 0;   // (nothing to place)
            continue;
        }
        char *base = (char *)B.arena;
        if (J.lgx >= 0) B.xs[B.lgx = J.lgx] = (uint4 *)(base + o_xs);
        BlockDev &D = b[j].dev;
        D.ptr = B.ptr = (const u32 *)(base + o_ptr);
        D.row = B.row = (const u32 *)(base + o_row);
        D.chunk = B.chunk = (const uint4 *)(base + o_chunk);
        D.lrow = B.lrow = (const u32 *)(base + o_lrow);
        D.col = B.col = (const u32 *)(base + o_col);
        D.val = B.val = base + o_val;
        D.carry = B.carry = (u64 *)(base + o_carry);
        D.count = B.count = (u32 *)(base + o_count);
        D.ncols = B.ncols;
        for (int c = 0; c <= kBlockClasses; ++c) D.row0[c] = (u32)B.cls_row[c];
        D.nchunk = (u32)B.nchunk;
        D.quad1 = B.quad1;
        D.small = b[j].small;
        D.fold = m <= (1u << 31) ? 1 : 0;
        D.M = make_mod(m, 1, 0);
        B.dev = (const BlockDev *)(base + o_dev);
        b[j].dev_out = (BlockDev *)(base + o_dev);
        b[j].optr = (u32 *)(base + o_ptr);
        b[j].orow = (u32 *)(base + o_row);
        b[j].chunk = (uint4 *)(base + o_chunk);
        b[j].lrow = (u32 *)(base + o_lrow);
        b[j].ocol = (u32 *)(base + o_col);
        b[j].oval = base + o_val;
        b[j].rows = (u32)rows;
        b[j].quads = (u32)quads;
    }
    memcpy(up.data(), b.data(), sizeof(BlockBuild) * b.size());
    memcpy(up.data() + o_cur, curs.data(), sizeof(u64) * curs.size());
    FF_CUDA(cudaMemcpyAsync(t, up.data(), head, cudaMemcpyHostToDevice, st));
    k_block_place<<<grid, kBlockThreads, 0, st>>>(dj, 1);
    k_block_fill<<<grid, kBlockThreads, 0, st>>>(dj);
    FF_CUDA(cudaGetLastError());
    FF_CUDA(cudaStreamSynchronize(st));
    return FFSPMV_OK;
}

// The jobs' layouts; every job's status, and that of its plan, set.
void run_jobs(BlockJob *jobs, int count)
{
    for (int j = 0; j < count; ++j) jobs[j].st = FFSPMV_OK;
    try {
        BlockScope S;
        const ffspmv_status r = build_blocks(jobs, count, S);
        for (int j = 0; j < count && r != FFSPMV_OK; ++j) jobs[j].st = r;
    } catch (const std::exception &) {
        for (int j = 0; j < count; ++j) jobs[j].st = FFSPMV_ERR_OOM;
    }
    for (int j = 0; j < count; ++j) {
        BlockPlan &B = *jobs[j].B;
        B.ok = jobs[j].st == FFSPMV_OK;
        B.memory.short_of = jobs[j].st == FFSPMV_ERR_OOM;
        if (B.ok || !B.arena) continue;
        cudaFree(B.arena);
        B.arena = nullptr;
        B.xs[B.lgx < 0 ? 0 : B.lgx] = nullptr;
        B.lgx = -1;
    }
}

}  // namespace

// A new plan for the job and whether it may be made; false without host memory.
static bool block_job(BlockJob &J, const ffspmv_handle *h, bool transpose, bool odd, int lgx)
{
    J = {new (std::nothrow) BlockPlan(), h, transpose, odd, lgx, FFSPMV_OK};
    if (!J.B) return false;
    try {
        J.st = block_limits(J);
    } catch (const std::exception &) {
        J.st = FFSPMV_ERR_OOM;
    }
    // testing: the first attempt finds no memory
    if (!odd && (h->opt.test_hooks & 16) && !h->block[transpose ? 1 : 0]) J.st = FFSPMV_ERR_OOM;
    J.B->memory.short_of = J.st == FFSPMV_ERR_OOM;
    return true;
}

ffspmv_status make_block(const ffspmv_handle *h, bool transpose, bool odd, int lgx, cudaStream_t st, BlockPlan **out)
{
    *out = nullptr;
    if (capturing(st)) return FFSPMV_ERR_CUDA;  // nothing can be allocated or copied now
    BlockJob J;
    if (!block_job(J, h, transpose, odd, lgx)) return FFSPMV_ERR_OOM;
    if (J.st == FFSPMV_OK) run_jobs(&J, 1);
    *out = J.B;
    return J.st;
}

void block_handles(int more)
{
    BlockKeep &K = block_keep();
    std::lock_guard<std::mutex> state(K.state);
    K.handles += more;
    if (K.handles) return;
    // no handle, so no build
    if (K.buf) cudaFreeHost(K.buf);
    K.buf = nullptr;
    for (cudaMemPool_t &p : K.pool) {
        if (p) cudaMemPoolDestroy(p);
        p = nullptr;
    }
}

void free_block_plan(BlockPlan *b)
{
    if (!b) return;
    if (b->arena) cudaFree(b->arena);
    for (int k = 0; k < kBlockStagings; ++k)
        if (b->xs[k] && k != b->lgx) cudaFree(b->xs[k]);
    delete b;
}

// Is a layout to be made (again)?
static bool block_wanted(BlockPlan *b) { return !b || (!b->ok && b->memory.again()); }

static void block_install(BlockPlan *&b, BlockPlan *made)
{
    if (b) made->memory.next(b->memory);
    free_block_plan(b);
    b = made;
}

BlockPlan *ensure_block(ffspmv_handle *h, bool transpose, const u32 *x, long long ldx, int nvec, cudaStream_t st)
{
    BlockPlan *&b = h->block[transpose ? 1 : 0];
    if (block_wanted(b)) {   // else it is there, cannot be made, or found no memory a while ago
        BlockPlan *made = nullptr;
        make_block(h, transpose, false, nvec ? staging_width(h->m <= 65536u, x, ldx, nvec) : -1, st, &made);
        if (made) block_install(b, made);
    }
    return b && b->ok ? b : nullptr;
}

void ensure_blocks(int count, ffspmv_handle *const *hs, const u32 *const *x, const int *nvec, cudaStream_t st)
{
    // builds share a stream and two waits, as many as fit this much temporary
    // memory: the first batch over 48 handles of 200 to 5 000 rows takes 11.6 ms
    // with a build each, 1.9 so
    constexpr size_t kTogether = (size_t)64 << 20;
    if (capturing(st)) return;
    std::vector<BlockJob> jobs;
    auto build = [&] {
        std::vector<BlockJob> go;
        for (const BlockJob &J : jobs)
            if (J.st == FFSPMV_OK) go.push_back(J);
        if (!go.empty()) run_jobs(go.data(), (int)go.size());
        for (BlockJob &J : go)
            if (go.size() > 1 && J.st == FFSPMV_ERR_OOM) run_jobs(&J, 1);   // not all at once, then
        for (BlockJob &J : jobs) block_install(const_cast<ffspmv_handle *>(J.h)->block[0], J.B);
        jobs.clear();
    };
    size_t bytes = 0;
    for (int i = 0; i < count; ++i) {
        ffspmv_handle *h = hs[i];
        if (!block_wanted(h->block[0])) continue;
        BlockJob J;
        if (!block_job(J, h, false, false, staging_width(h->m <= 65536u, x[i], nvec[i], nvec[i]))) continue;
        const size_t more = block_job_bytes(J);
        if (!jobs.empty() && (bytes + more > kTogether || jobs.size() >= 1024)) {
            build();
            bytes = 0;
        }
        bytes += more;
        jobs.push_back(J);
    }
    build();
}

std::string block_summary(const BlockPlan *b)
{
    if (!b || !b->ok) return "";
    size_t staged = 0;
    for (int k = 0; k < kBlockStagings; ++k)
        if (b->xs[k]) staged += ((size_t)b->ncols << k) * sizeof(uint4);
    char buf[160];
    snprintf(buf, sizeof buf, "  blocks: rows in length classes, %lld in %lld chunks, %s values, %zu bytes of staged rows of X\n",
             b->nlong, b->nchunk, b->small ? "u16" : "u32", staged);
    return buf;
}

// The staging buffer for 2^lg pieces per row.
static uint4 *block_buffer(BlockPlan &B, int lg, cudaStream_t st)
{
    for (int k = lg; k < kBlockStagings; ++k)
        if (B.xs[k]) return B.xs[k];
    if (capturing(st) || (B.staging.short_of && !B.staging.again())) return nullptr;
    BlockScope S;   // (another stream may be under capture)
    if (cudaMalloc((void **)&B.xs[lg], ((size_t)B.ncols << lg) * sizeof(uint4)) != cudaSuccess) {
        cudaGetLastError();
        B.xs[lg] = nullptr;
        B.staging.next(B.staging);
        B.staging.short_of = true;
        return nullptr;
    }
    B.staging = BlockMemory();
    return B.xs[lg];
}

bool block_staging(BlockPlan &B, const u32 *x, long long ldx, int nvec, cudaStream_t st, uint4 **xs)
{
    const int lg = staging_width(B.small, x, ldx, nvec);
    *xs = lg < 0 || B.ncols == 0 ? nullptr : block_buffer(B, lg, st);
    return lg < 0 || B.ncols == 0 || *xs;
}

int block_pieces(const BlockPlan &B, const u32 *x, int nvec)
{
    const int C = B.small ? 8 : 4;
    return block_in_place(B.small, x, nvec, nvec) || B.ncols == 0 ? 0 : (nvec + C - 1) / C;
}

uint4 *block_staging(BlockPlan &B, int most, int total, cudaStream_t st, int *room)
{
    constexpr long long kWords = (64LL << 20) / sizeof(uint4);   // and 64 MB, or one block's
    const int want = (int)std::max<long long>(most, std::min<long long>(std::min(total, kBlockPieces), kWords / B.ncols));
    for (int p : {want, most}) {
        int lg = 0;
        while ((1 << lg) < p) ++lg;
        if (uint4 *xs = block_buffer(B, lg, st)) {
            *room = 1 << lg;
            return xs;
        }
    }
    return nullptr;
}

long long block_launches(const BlockPlan &B, int nvec)
{
    long long n = 0;
    for (int v0 = 0; v0 < nvec; v0 += kBlockVecs)
        n += block_in_place(B.small, nullptr, nvec, std::min(kBlockVecs, nvec - v0)) ? 1 : 2;
    return n;
}

// What a launch needs of the layout and of one block of nv vectors (X is
// filled in by the caller).
static BlockArgs block_args(const BlockPlan &B, u32 *y, long long ldy, int nv, u32 m, u32 alpha, u32 beta)
{
    BlockArgs a;
    memset(&a, 0, sizeof(a));
    a.m.ptr = B.ptr;
    a.m.row = B.row;
    a.m.col = B.col;
    a.m.lrow = B.lrow;
    a.m.chunk = B.chunk;
    a.m.val = B.val;
    a.m.carry = B.carry;
    a.m.count = B.count;
    a.m.quad1 = B.quad1;
    a.m.y = y;
    a.m.ldy = ldy;
    a.m.nvec = nv;
    a.m.vec4 = (ldy % 4 == 0 && ((uintptr_t)y & 15u) == 0) ? 1 : 0;
    a.m.M = make_mod(m, alpha, beta);
    a.m.fold = m <= (1u << 31) ? 1 : 0;
    const int C = B.small ? 8 : 4;
    a.m.pieces = (nv + C - 1) / C;
    while ((1 << a.m.lgt) < a.m.pieces) ++a.m.lgt;
    return a;
}

// The warps of a launch, class by class; returns their number.
static long long block_warps(const BlockPlan &B, BlockArgs &a)
{
    // groups per row: by class, doubled while the launch has fewer than
    // 16 warps per SM (short matrices: more lanes per row, shorter chains)
    long long warps = 0;
    for (int boost = 0; boost < 6; ++boost) {
        warps = B.nchunk;
        for (int c = 0; c < kBlockClasses; ++c) {
            const int lg = std::min(block_lgg(c, a.m.lgt) + boost, 5 - a.m.lgt);
            a.lgg[c] = lg;
            a.row0[c] = (u32)B.cls_row[c];
            a.warp0[c] = (u32)warps;
            const int rpw = 32 >> (a.m.lgt + lg);
            warps += (B.cls_row[c + 1] - B.cls_row[c] + rpw - 1) / rpw;
        }
        if (warps >= 16LL * B.nsm) break;
    }
    a.row0[kBlockClasses] = (u32)B.cls_row[kBlockClasses];
    a.warp0[kBlockClasses] = (u32)warps;
    a.nchunk_warps = (int)B.nchunk;
    return warps;
}

ffspmv_status run_block(const BlockPlan &B, uint4 *xs, const u32 *x, long long ldx, u32 *y, long long ldy, int nvec,
                        u32 m, u32 alpha, u32 beta, cudaStream_t st)
{
    const int C = B.small ? 8 : 4;
    for (int v0 = 0; v0 < nvec; v0 += kBlockVecs) {
        const int nv = std::min(kBlockVecs, nvec - v0);
        const u32 *xv = x + v0;
        u32 *yv = y + v0;
        BlockArgs a = block_args(B, yv, ldy, nv, m, alpha, beta);
        const int pieces = (nv + C - 1) / C;
        const bool in_place = block_in_place(B.small, xv, ldx, nv);
        if (in_place) {
            a.m.xs = reinterpret_cast<const uint4 *>(xv);
            a.m.pitch = (int)(ldx / 4);
        } else {
            a.m.xs = xs;
            a.m.pitch = pieces;
            const long long words = B.ncols * pieces;
            const int vec4 = (ldx % 4 == 0 && ((uintptr_t)xv & 15u) == 0) ? 1 : 0;
            if (words > 0) {
                const unsigned blocks = (unsigned)((words + kBlockThreads - 1) / kBlockThreads);
                if (B.small)
                    k_block_stage<true><<<blocks, kBlockThreads, 0, st>>>(xv, ldx, B.ncols, nv, pieces, vec4, xs);
                else
                    k_block_stage<false><<<blocks, kBlockThreads, 0, st>>>(xv, ldx, B.ncols, nv, pieces, vec4, xs);
                FF_CUDA(cudaGetLastError());
            }
        }
        const long long warps = block_warps(B, a);
        if (warps == 0) continue;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((warps * 32 + kBlockThreads - 1) / kBlockThreads));
        cfg.blockDim = dim3(kBlockThreads);
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = in_place ? 0 : 1;
        if (B.small) FF_CUDA(cudaLaunchKernelEx(&cfg, k_block<true>, a));
        else FF_CUDA(cudaLaunchKernelEx(&cfg, k_block<false>, a));
    }
    return FFSPMV_OK;
}

// Y_j = A_j X_j for `count` (at most kMany) different plans, contiguous blocks
// of nvec[j] <= kBlockVecs vectors.
static ffspmv_status block_many(int count, const BlockPlan *const *B, uint4 *const *xs, const u32 *const *x, u32 *const *y,
                                const int *nvec, const int *v0, cudaStream_t st)
{
    BlockMany P, S;   // the products, and the staging of the X that are not read in place
    memset(&P, 0, sizeof(P));
    memset(&S, 0, sizeof(S));
    long long warps = 0, stage = 0;
    for (int j = 0; j < count; ++j) {
        const BlockPlan &b = *B[j];
        const int C = b.small ? 8 : 4, pieces = (nvec[j] + C - 1) / C;
        int lgt = 0;
        while ((1 << lgt) < pieces) ++lgt;
        P.dev[j] = b.dev;
        const bool place = block_in_place(b.small, x[j], nvec[j], nvec[j]);
        P.x[j] = x[j];
        P.xs[j] = xs[j];
        P.y[j] = y[j];
        P.nvec[j] = (unsigned char)(nvec[j] | (place ? 128 : 0));
        P.v0[j] = (unsigned char)v0[j];
        P.first[j] = (u32)warps;
        warps += b.nchunk;
        for (int c = 0; c < kBlockClasses; ++c) {
            const int rpw = 1 << (5 - lgt - block_lgg(c, lgt));
            warps += (b.cls_row[c + 1] - b.cls_row[c] + rpw - 1) / rpw;
        }
        if (!place && b.ncols > 0) {
            S.dev[S.count] = b.dev;
            S.x[S.count] = x[j];
            S.xs[S.count] = xs[j];
            S.nvec[S.count] = (unsigned char)nvec[j];
            S.first[S.count++] = (u32)stage;
            stage += (b.ncols * pieces + kBlockThreads - 1) / kBlockThreads;
        }
    }
    if (warps >= (1LL << 32) - 64 || stage >= (1LL << 31)) return FFSPMV_ERR_UNSUPPORTED;
    P.first[count] = (u32)warps;
    P.count = count;
    if (stage > 0) {
        S.first[S.count] = (u32)stage;
        k_block_stage_many<<<(unsigned)stage, kBlockThreads, 0, st>>>(S);
        FF_CUDA(cudaGetLastError());
    }
    if (warps == 0) return FFSPMV_OK;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((warps * 32 + kBlockThreads - 1) / kBlockThreads));
    cfg.blockDim = dim3(kBlockThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = stage > 0 ? 1 : 0;
    FF_CUDA(cudaLaunchKernelEx(&cfg, k_block_many, P));
    return FFSPMV_OK;
}

ffspmv_status run_block_many(int count, const BlockPlan *const *B, uint4 *const *xs, const u32 *const *x, u32 *const *y,
                             const int *nvec, const int *v0, cudaStream_t st)
{
    for (int c0 = 0; c0 < count; c0 += kMany) {
        const ffspmv_status r =
            block_many(std::min(kMany, count - c0), B + c0, xs + c0, x + c0, y + c0, nvec + c0, v0 + c0, st);
        if (r != FFSPMV_OK) return r;
    }
    return FFSPMV_OK;
}

// projecting CTAs: four rows per group of threads, two CTAs per SM at most
static unsigned step_proj(long long n, int s)
{
    const int ngrp = kBlockThreads / (s * ((s + 3) / 4));
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return (unsigned)std::max<long long>(1, std::min<long long>((n + 4LL * ngrp - 1) / (4LL * ngrp), 2LL * std::max(nsm, 1)));
}

size_t block_steps_bytes(long long n, int s) { return (size_t)2 * step_proj(n, s) * s * s * 4; }

ffspmv_status run_block_steps(const BlockPlan &B, long long n, int s, u32 m, const u32 *X, u32 *V0, u32 *V1, u32 *part,
                              long long nsteps, bool next, u32 *S, cudaStream_t st)
{
    const int ldv = (s + 3) / 4 * 4;
    BlockStep a;
    memset(&a, 0, sizeof(a));
    a.s = s;
    a.tiles = s * (ldv / 4);
    a.ngrp = kBlockThreads / a.tiles;
    a.n = n;
    a.ldv = ldv;
    a.X = X;
    a.proj = step_proj(n, s);
    a.fin = (unsigned)((s * s + kStepOuts - 1) / kStepOuts);
    a.per = (n + a.proj - 1) / a.proj;
    u32 *parts[2] = {part, part + (size_t)a.proj * s * s};
    for (long long i = 0; i <= nsteps; ++i) {
        const u32 *Vi = (i & 1) ? V1 : V0;
        a.b = block_args(B, (i & 1) ? V0 : V1, ldv, s, m, 1, 0);
        a.b.m.xs = reinterpret_cast<const uint4 *>(Vi);
        a.b.m.pitch = ldv / 4;
        const long long warps = block_warps(B, a.b);
        a.spmm = i + 1 < nsteps || (next && i < nsteps) ? (unsigned)((warps * 32 + kBlockThreads - 1) / kBlockThreads) : 0u;
        a.V = Vi;
        a.part = parts[i & 1];
        a.prev = i ? parts[(i + 1) & 1] : nullptr;
        a.S = i ? S + (i - 1) * s * s : nullptr;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(a.spmm + (i < nsteps ? a.proj : 0u) + a.fin);
        cfg.blockDim = dim3(kBlockThreads);
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        FF_CUDA(cudaLaunchKernelEx(&cfg, k_block_step, a));
    }
    return FFSPMV_OK;
}

}  // namespace ff
