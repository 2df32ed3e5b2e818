// Sigma-bases over F_p for the second step of block Wiedemann (Sec. 3.2,
// "Parallelization of the sigma-basis computation"): PM-Basis (Giorgi,
// Jeannerod and Villard, ISSAC 2003) as a host recursion on the order whose
// work is polynomial-matrix products on the GPU (polymat.cu, Sec. 3.2.1's
// evaluation / pointwise / interpolation scheme, and products by definition
// for short operands), and M-Basis, the iterative algorithm Sec. 3.2.2
// recommends at small orders, as one CTA per leaf.
//
// The recursion.  An order-d basis is P2 P1 with P1 of order d1 = ceil(d/2)
// and P2 of the residual, the coefficients d1..d-1 of P1 F, with P1's degrees
// as its shift.  M-Basis itself is the recursion's limit (order k's operations
// depend only on that order's residual and the current degrees), so the
// result is the same matrix wherever the leaves are cut; the leaves here take
// at most kSbLeaf orders.  Up to order kSbAsync a node needs nothing from the
// host: degrees and degree bounds stay in device slots, the products are
// direct (one launch each) and the launches queue up.  Above it the host
// reads each half's degree bound to size the transforms, of exactly the
// coefficients that are needed: the residual is a middle product whose cyclic
// wrap falls on coefficients below d1.
//
// M-Basis leaf.  Order k eliminates R_k (m x n) column by column: rows
// ordered by (delta_i, i), the pivot the first non-pivot row nonzero in the
// column, multiples of it added to later rows, then the pivot rows times x.
// The elimination is fraction free (row r becomes a r - b q), so no inverse
// is taken inside the loop; one inversion per row at the end of the leaf
// divides out its multipliers, which makes the result the plain algorithm's.
// It is the serial part: four warps of the leaf's first CTA do nothing else,
// a lane per row in pivot order, a panel of a quarter of the columns each in
// registers.  Panel by panel, its owner shares the panel's columns, and every
// warp eliminates them (the same few operations, redundantly) while it applies
// each step to its own columns, so that a step needs no exchange between
// warps.  Nearly always the pivots are the rows in order, so a panel first
// takes them as known: a step is then a shuffle and a multiply-add long, with
// no vote on the way; it is done again with votes if one of them turns out
// zero.  A column's register turns from R_k's entry into the coefficient of
// its pivot once its step is done, so what comes out is a matrix: every row
// becomes c r plus a combination of the *original* pivot rows.  Eight other
// warps apply it to R's later coefficients as independent multiply-adds, the
// coefficient that the next elimination waits for first; two more CTAs of
// the cluster, which get the matrix through distributed shared memory, apply
// it to P.
//
// What bounds it: 64-bit multiply-adds, at 32 per clock and SM, and the chain
// of n dependent steps.  One order of R and P (about 7 500 clocks of one SM
// at order 16, 32 x 16) is therefore spread over three SMs and mostly off the
// elimination's path (about 180 clocks per step).  Measured, order 12 502,
// 32 x 16, p = 65521: one cluster of eight CTAs per leaf of order 24-25 that
// exchanged every row operation took about 20 us per order and 293 ms for
// the whole basis (with the transforms of polymat.cu); one warp eliminating
// beside sixteen that apply, on one SM, 10 us; four warps and three CTAs, a
// vote and an exchange per column, 5.7 us (98 ms); as it is here 4.4 us and
// 81 ms.
#include <algorithm>
#include <climits>
#include <cstddef>
#include <cstring>
#include <vector>

#include "ff_internal.cuh"
#include "ff_polymat.h"
#include "ffspmv_polymat.h"
#include "ffspmv_sigma.h"

namespace ff {
namespace {

constexpr int kSbMaxM = 32;                 // rows of F and of P (the polynomial-matrix product's limit)
constexpr int kSbMaxBase = 32;              // largest leaf order a caller may name
constexpr int kSbLeaf = 16;                 // largest order of one M-Basis launch
constexpr long long kSbAsync = 200;         // largest order whose nodes run without the host
constexpr int kSbUpd = 16;                  // warps that apply the operations
constexpr int kSbElim = 4;                  // warps that eliminate (first CTA)
constexpr int kSbRes = 8;                   // of kSbUpd, in the first CTA: two per scheduler, which each leave it to its eliminating warp most of the time
constexpr int kSbFirst = 32 * (kSbRes + kSbElim);   // threads that work in the first CTA
constexpr int kSbThreads = 32 * (kSbUpd + kSbElim);
constexpr int kSbCtas = 3;                  // the first CTA: elimination and R; the others: P
constexpr size_t kSbSmemMax = 227 * 1024;
constexpr size_t kSbAlign = 256;
constexpr int kSbMaxShift = 1 << 24;

struct SbLeaf {
    const u32 *F;        // d x m x n residues
    u32 *P;              // out: (d+1) x m x m
    const int *shift;    // m
    SbSlot *out;
    int m, n, d;
    int rs, ps;          // words per row of R and of P in shared memory
    u32 pinv;            // p^-1 mod 2^32 (odd p)
    Mod M;
};

// Shared memory of a leaf's CTA: the operations of an order (two copies, by
// order parity), the final row scales, the elimination's exchange; then in
// the first CTA R twice (an order reads one copy and writes the other), in
// the others P, row by row: word t n4 + c of a row of R is coefficient t,
// column c (n4 = n rounded up to 4), the same for P with m4.  Row strides are
// 4 mod 32 words: the rows a quarter warp reads 16 bytes from lie in distinct
// banks.
struct SbOps {
    u32 T[kSbMaxM][kSbMaxM];   // [column][row]: what row gets of the column's pivot row
    u32 c[kSbMaxM];            // [row]: what it keeps of itself
    u32 q[kSbMaxM];            // [column]: byte offset of the pivot row (any row, with T = 0, when there is none)
    u32 qp[kSbMaxM];           // [column]: the same offset in P
    int isp[kSbMaxM];          // [row]: 1 for the pivot rows
};
typedef u32 SbPanel[2][8][32];   // a panel's columns, by lane of the eliminating warps; two copies
constexpr size_t kSbOpsBytes = sizeof(SbOps);
constexpr size_t kSbScaleOff = 2 * kSbOpsBytes;
constexpr size_t kSbOrdOff = kSbScaleOff + kSbMaxM * 4;                 // [kSbElim][32]
constexpr size_t kSbXOff = kSbOrdOff + kSbElim * 32 * 4;                // SbPanel
constexpr size_t kSbRowOff = kSbXOff + sizeof(SbPanel);
static_assert(kSbRowOff % 16 == 0, "16-byte rows");

int sb_stride(int words) { return (words + 27) / 32 * 32 + 4; }
int sb_rstride(int n, long long d) { return sb_stride((int)d * ((n + 3) / 4 * 4)); }
int sb_pstride(int m, long long d) { return sb_stride((int)(d + 1) * ((m + 3) / 4 * 4)); }

size_t sb_leaf_smem(int m, int n, long long d)
{
    return kSbRowOff + (size_t)std::max(2 * sb_rstride(n, d), sb_pstride(m, d)) * m * 4;
}

__device__ u32 sb_pow(u32 a, u32 e, const Mod &M)
{
    u32 r = 1u % M.m;
    while (e) {
        if (e & 1u) r = red64((u64)r * a, M);
        a = red64((u64)a * a, M);
        e >>= 1;
    }
    return r;
}

// x 2^-32 mod p for x < p 2^32 (Montgomery, 1985), in [0, p).  p = 2 has no
// inverse mod 2^32: there x mod p, without the factor; the factor scales
// rows, and the row scales are kept by this same function.
template <bool EVEN>
__device__ __forceinline__ u32 sb_red(u64 x, const SbLeaf &a)
{
    if constexpr (EVEN) return red64(x, a.M);
    const u32 p = a.M.m, r = (u32)(x >> 32) + p - __umulhi((u32)x * a.pinv, p);
    return min(r, r - p);
}

__device__ __forceinline__ u64 sb_fold(u64 x, u32 p)   // x < 2 p 2^32 -> x mod p 2^32
{
    const u32 h = (u32)(x >> 32);
    return (u64)min(h, h - p) << 32 | (u32)x;
}

// The shared::cluster address of `local` in CTA `rank` of the cluster.
__device__ __forceinline__ u32 sb_remote(const void *local, u32 rank)
{
    u32 r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((u32)__cvta_generic_to_shared(local)), "r"(rank));
    return r;
}

__device__ __forceinline__ void sb_st_remote(u32 addr, u32 v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void sb_st_remote_v4(u32 addr, uint4 v)
{
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

__device__ __forceinline__ void sb_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// ... by a thread whose writes no other CTA reads
__device__ __forceinline__ void sb_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void sb_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ u32 sb_rank()
{
    u32 r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// The operations applied to W (1 or 2) adjacent columns of one coefficient:
// lane r gets row r's new values.  `row0` points at the columns in row 0.
// FOLD (p > 2^26): two products below p^2 are added to a sum below p 2^32,
// then the sum is brought back below that; else all 33 fit.
template <int W>
struct SbVec;
template <>
struct SbVec<1> {
    typedef u32 V;
    static __device__ __forceinline__ u32 get(u32 v, int) { return v; }
};
template <>
struct SbVec<2> {
    typedef uint2 V;
    static __device__ __forceinline__ u32 get(const uint2 &v, int i) { return i ? v.y : v.x; }
};

template <class V>
__device__ __forceinline__ V sb_at(const u32 *row0, u32 bytes)
{
    return *reinterpret_cast<const V *>(reinterpret_cast<const char *>(row0) + bytes);
}

// The offsets of the pivot rows: in registers while there is room for them.
template <int N>
struct SbPiv {
    u32 q[N <= 16 ? N : 1];
    const u32 *s;
    __device__ __forceinline__ SbPiv(const u32 *sm) : s(sm)
    {
        if constexpr (N <= 16) {
#pragma unroll
            for (int j = 0; j < N; j += 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(sm + j);
                q[j] = v.x; q[j + 1] = v.y; q[j + 2] = v.z; q[j + 3] = v.w;
            }
        }
    }
    __device__ __forceinline__ u32 at(int j) const
    {
        if constexpr (N <= 16) return q[j];
        else return s[j];
    }
};

// All N columns, without a branch on n: columns without a pivot bring T = 0
// and the loads of all the pivot rows are in flight together.
template <int N, int W, bool FOLD, bool EVEN>
__device__ __forceinline__ void sb_apply(u32 (&out)[W], const SbLeaf &a, const u32 *row0, u32 own_off, const SbPiv<N> &Q, u32 c,
                                         const u32 (&T)[N])
{
    typedef typename SbVec<W>::V V;
    const u32 p = a.M.m;
    const V own = sb_at<V>(row0, own_off);
    u64 x[W];
#pragma unroll
    for (int i = 0; i < W; ++i) x[i] = (u64)c * SbVec<W>::get(own, i);
#pragma unroll
    for (int j = 0; j < N; j += 2) {
        const V v0 = sb_at<V>(row0, Q.at(j)), v1 = sb_at<V>(row0, Q.at(j + 1));
#pragma unroll
        for (int i = 0; i < W; ++i) {
            x[i] += (u64)T[j] * SbVec<W>::get(v0, i);
            x[i] += (u64)T[j + 1] * SbVec<W>::get(v1, i);
            if (FOLD) x[i] = sb_fold(x[i], p);
        }
    }
#pragma unroll
    for (int i = 0; i < W; ++i) out[i] = sb_red<EVEN>(x[i], a);
}

// N: 8, 16 or 32, at least n.  One cluster of kSbCtas CTAs.  The cluster
// barrier has one phase per order: a thread of the first CTA arrives once
// order k's operations are in every CTA and waits before the next order's are
// written; one of the others arrives when it is done with order k - 1 and
// waits for order k's operations.
template <int N, bool FOLD, bool EVEN>
__global__ void __launch_bounds__(kSbThreads, 1) k_sb_mbasis(const __grid_constant__ SbLeaf a)
{
    extern __shared__ __align__(16) unsigned char sb_sm[];
    const int m = a.m, n = a.n, d = a.d;
    const u32 p = a.M.m;
    const int n4 = (n + 3) & ~3, m4 = (m + 3) & ~3;
    SbOps *ops = reinterpret_cast<SbOps *>(sb_sm);
    u32 *scale = reinterpret_cast<u32 *>(sb_sm + kSbScaleOff);
    u32 *rows = reinterpret_cast<u32 *>(sb_sm + kSbRowOff);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const u32 cta = sb_rank();

    for (int i = tid; i < (int)(2 * kSbOpsBytes / 4); i += kSbThreads) reinterpret_cast<u32 *>(ops)[i] = 0u;
    const int words = (cta == 0 ? 2 * a.rs : a.ps) * m;
    for (int i = tid; i < words; i += kSbThreads) rows[i] = 0u;
    __syncthreads();
    if (cta == 0) {
        for (int i = tid; i < d * m * n; i += kSbThreads) {
            const int c = i % n, tr = i / n, t = tr / m, r = tr - t * m;
            rows[r * a.rs + t * n4 + c] = __ldg(a.F + i);
        }
    } else if (tid < m) {
        rows[tid * a.ps + tid] = 1u;   // P = identity
    }
    __syncthreads();
    sb_arrive();
    sb_wait();   // every CTA's operations are cleared before any remote store

    if (cta == 0 && warp >= kSbUpd) {
        // the eliminating warps: each keeps row r's degree and scale in lane r
        constexpr int NC = N / kSbElim;   // columns per warp: ew NC ...
        const int ew = warp - kSbUpd, col0 = ew * NC;
        int *ord = reinterpret_cast<int *>(sb_sm + kSbOrdOff) + ew * 32;
        auto &X = *reinterpret_cast<SbPanel *>(sb_sm + kSbXOff);
        int dl = lane < m ? __ldg(a.shift + lane) : INT_MAX;
        int smin = dl;
        u32 tot = 1u;
        for (int k = 0; k < d; ++k) {
            // lane 31 - l takes the row of rank l in the order (delta, index),
            // so that the first candidate of a vote is its highest bit.  Rows
            // of one delta at a time: generic inputs have two or three values
            int rank = 31;
            for (u32 left = 0xffffffffu; left;) {   // warp-uniform
                const int v = __reduce_min_sync(0xffffffffu, (left >> lane) & 1u ? dl : INT_MAX);
                const u32 same = __ballot_sync(0xffffffffu, ((left >> lane) & 1u) && dl == v);
                if ((left >> lane) & 1u) rank -= dl == v ? __popc(same & ((1u << lane) - 1u)) : __popc(same);
                left &= ~same;
            }
            __syncwarp();
            ord[rank] = lane;
            __syncwarp();
            const int row = ord[lane];
            const bool live = row < m;
            // R_k, once the other warps have it
            if (k) asm volatile("bar.sync 1, %0;" ::"n"(kSbFirst) : "memory");
            u32 R[NC];
            const u32 *src = rows + (k & 1) * (a.rs * m) + (live ? row : 0) * a.rs + k * n4 + col0;
#pragma unroll
            for (int s = 0; s < NC; ++s) R[s] = live && col0 + s < n ? src[s] : 0u;
            u32 c = 1u;
            bool isp = false;
            int q_of = 31;   // lane j: lane of column j's pivot row (31: the first row, for columns without one)
#pragma unroll
            for (int w = 0; w < kSbElim; ++w) {
                if (w * NC < n) {
                    const bool mine = ew == w;
                    u32 *xs = &X[w & 1][0][0];
                    if (mine) {
#pragma unroll
                        for (int j = 0; j < NC; ++j) xs[j * 32 + lane] = R[j];
                    }
                    asm volatile("bar.sync 3, %0;" ::"n"(kSbElim * 32) : "memory");
                    u32 pc[NC];   // the panel's columns
#pragma unroll
                    for (int j = 0; j < NC; ++j) pc[j] = xs[j * 32 + lane];
                    // step j with pivot lane q: row <- av row - x pivot row
                    // (times 2^-32) for the rows in `act`; the others compute
                    // it too and drop it.  The panel's next column first: the
                    // next step waits for it
                    auto step = [&](int j, int q, bool act, u32 av) {
                        const u32 g = p - pc[j];
#pragma unroll
                        for (int i = 0; i < NC; ++i) {
                            if (i > j) {
                                const u32 o = __shfl_sync(0xffffffffu, pc[i], q);
                                const u32 v = sb_red<EVEN>((u64)av * pc[i] + (u64)g * o, a);
                                pc[i] = act ? v : pc[i];
                            }
                        }
                        const u32 cq = __shfl_sync(0xffffffffu, c, q);
#pragma unroll
                        for (int i = 0; i < NC; ++i) {
                            // the owner's column j is done: the coefficient of its pivot begins
                            const bool here = mine && i == j;
                            const u32 old = here ? 0u : R[i], o = __shfl_sync(0xffffffffu, R[i], q);
                            const u32 v = sb_red<EVEN>((u64)av * old + (u64)g * (here ? cq : o), a);
                            R[i] = act ? v : old;
                        }
                        const u32 cv = sb_red<EVEN>((u64)av * c, a);
                        c = act ? cv : c;
                    };
                    // first with the rows in order as pivots, lanes 31 - w NC,
                    // 30 - w NC ..: right if the panels before took the lanes
                    // above and no pivot is zero
                    const u32 above = w == 0 ? 0u : ~0u << (32 - NC * w);
                    bool good = w * NC + NC <= n && __ballot_sync(0xffffffffu, isp) == above;
                    if (good) {
                        u32 keep[NC], z = 0xffffffffu;
                        const u32 ckeep = c;
#pragma unroll
                        for (int j = 0; j < NC; ++j) keep[j] = R[j];
#pragma unroll
                        for (int j = 0; j < NC; ++j) {
                            const int q = 31 - w * NC - j;
                            const u32 av = __shfl_sync(0xffffffffu, pc[j], q);
                            z = min(z, av);
                            step(j, q, lane < q, av);
                        }
                        good = z != 0u;
                        if (good) {
                            isp = lane >= 32 - w * NC - NC;
                            if (lane >= w * NC && lane < w * NC + NC) q_of = 31 - lane;
                        } else {
                            c = ckeep;
#pragma unroll
                            for (int j = 0; j < NC; ++j) {
                                R[j] = keep[j];
                                pc[j] = xs[j * 32 + lane];
                            }
                        }
                    }
                    if (!good) {
#pragma unroll
                        for (int j = 0; j < NC; ++j) {
                            const bool cand = !isp && pc[j] != 0u;
                            const u32 b = __ballot_sync(0xffffffffu, cand);
                            // (no candidate: the column is zero in every row left,
                            // nothing is taken over and the coefficients are 0)
                            const int q = b ? 31 - __clz(b) : 31;
                            step(j, q, cand && lane != q, __shfl_sync(0xffffffffu, pc[j], q));
                            isp = isp || (cand && lane == q);
                            if (lane == w * NC + j) q_of = q;
                        }
                    }
                }
            }
            SbOps &O = ops[k & 1];
            const int qrow = ord[q_of];   // always a row below m: candidates are, and so is the first in the order
            const u32 pb = __ballot_sync(0xffffffffu, isp);
            if (live) {
#pragma unroll
                for (int s = 0; s < NC; ++s) O.T[col0 + s][row] = R[s];
                if (ew == 0) O.c[row] = c;
                if (ew == 1) O.isp[row] = isp ? 1 : 0;
            }
            if (ew == 2) O.q[lane] = (u32)(qrow * a.rs * 4);
            if (ew == 3) O.qp[lane] = (u32)(qrow * a.ps * 4);
            // the operations of order k are complete: the other warps go on
            // (this one meets them again when it has to have R)
            asm volatile("bar.arrive 2, %0;" ::"n"(kSbThreads) : "memory");
            if (k) sb_wait();
            sb_arrive_relaxed();
            const u32 cr = __shfl_sync(0xffffffffu, c, rank);
            if (lane < m) {
                dl += (int)((pb >> rank) & 1u);
                tot = sb_red<EVEN>((u64)tot * cr, a);
            }
        }
        sb_wait();
        if (ew == 0) {
            const u32 inv = lane < m ? sb_pow(tot, p - 2u, a.M) : 0u;   // tot is not 0 in the field F_p
            for (u32 r = 1; r < kSbCtas; ++r) sb_st_remote(sb_remote(scale + lane, r), inv);
            int dmax = lane < m ? dl : INT_MIN;
            smin = __reduce_min_sync(0xffffffffu, smin);
            dmax = __reduce_max_sync(0xffffffffu, dmax);
            a.out->delta[lane] = lane < m ? dl : 0;
            if (lane == 0) {
                a.out->e = max(0, min(d, dmax - smin));
                a.out->smin = smin;
                a.out->dmax = dmax;
            }
        }
    } else if (cta == 0 && warp >= kSbRes) {
        // the warps between: an order's operations into the other CTAs, once
        // these read the operations of two orders ago no more
        for (int k = 0; k < d; ++k) {
            asm volatile("bar.sync 2, %0;" ::"n"(kSbThreads) : "memory");
            if (k) sb_wait();
            const uint4 *src = reinterpret_cast<const uint4 *>(&ops[k & 1]);
            for (int e = tid - 32 * kSbRes; e < (int)(kSbOpsBytes / 16); e += 32 * (kSbUpd - kSbRes)) {
                // columns past n of T stay zero everywhere
                if (e >= n * 8 && e < kSbMaxM * 8) continue;
                const uint4 v = src[e];
                for (u32 r = 1; r < kSbCtas; ++r) sb_st_remote_v4(sb_remote(src + e, r), v);
            }
            __syncwarp();
            sb_arrive();
        }
        sb_wait();
    } else if (cta == 0) {
        const int np = n4 / 2;   // column pairs of R
        for (int k = 0; k < d; ++k) {
            asm volatile("bar.sync 2, %0;" ::"n"(kSbThreads) : "memory");
            sb_arrive_relaxed();
            const SbOps &O = ops[k & 1];
            const u32 *R0 = rows + (k & 1) * (a.rs * m);
            u32 *R1 = rows + ((k + 1) & 1) * (a.rs * m);
            const u32 c = O.c[lane];
            const int up = O.isp[lane];   // pivot rows move up by one coefficient
            u32 T[N];
#pragma unroll
            for (int j = 0; j < N; ++j) T[j] = O.T[j][lane];
            const SbPiv<N> Q(O.q);
            const u32 own = (u32)(min(lane, m - 1) * a.rs * 4);
            auto r_unit = [&](const u32 *at, int t, int pr) {   // lane r: coefficient t of R, column pair pr, at `at`
                u32 v[2];
                sb_apply<N, 2, FOLD, EVEN>(v, a, at, own, Q, c, T);
                if (lane < m && t + up < d)
                    *reinterpret_cast<uint2 *>(R1 + lane * a.rs + (t + up) * n4 + 2 * pr) = make_uint2(v[0], v[1]);
            };
            if (k + 1 < d) {
                // coefficient k + 1 first: from k for the pivot rows, from k + 1 for the others
                for (int u = warp; u < np; u += kSbRes) r_unit(R0 + (k + 1 - up) * n4 + 2 * u, k + 1 - up, u);
                asm volatile("bar.arrive 1, %0;" ::"n"(kSbFirst) : "memory");
                // coefficients k + 1 (pivot rows: to k + 2) .. d - 1
                for (int pr = warp; pr < np; pr += kSbRes) {
                    u32 *to = R1 + lane * a.rs + 2 * pr;
                    for (int t = k + 1; t < d; ++t) {
                        u32 v[2];
                        sb_apply<N, 2, FOLD, EVEN>(v, a, R0 + t * n4 + 2 * pr, own, Q, c, T);
                        if (lane < m && t + up < d && t + up > k + 1)
                            *reinterpret_cast<uint2 *>(to + (t + up) * n4) = make_uint2(v[0], v[1]);
                    }
                }
            }
            sb_wait();
        }
    } else {
        // P in place: a column belongs to one warp, top coefficient first
        const int per = (kSbCtas - 1) * kSbUpd;
        for (int k = 0; k < d; ++k) {
            sb_arrive();
            sb_wait();
            if (warp >= kSbUpd) continue;
            const SbOps &O = ops[k & 1];
            const u32 c = O.c[lane];
            const int up = O.isp[lane];
            u32 T[N];
#pragma unroll
            for (int j = 0; j < N; ++j) T[j] = O.T[j][lane];
            const SbPiv<N> Q(O.qp);
            const u32 own = (u32)(min(lane, m - 1) * a.ps * 4);
            for (int w = ((int)cta - 1) * kSbUpd + warp; w < m; w += per) {
                u32 *at = rows + k * m4 + w, *to = at + lane * a.ps + up * m4;
                int t = k;
                for (; t > 0; t -= 2, at -= 2 * m4, to -= 2 * m4) {   // two coefficients at a time
                    u32 v[1], u[1];
                    sb_apply<N, 1, FOLD, EVEN>(v, a, at, own, Q, c, T);
                    sb_apply<N, 1, FOLD, EVEN>(u, a, at - m4, own, Q, c, T);
                    __syncwarp();   // every lane has read them
                    if (lane < m) {
                        to[0] = v[0];
                        to[-m4] = u[0];
                    }
                }
                if (t == 0) {
                    u32 v[1];
                    sb_apply<N, 1, FOLD, EVEN>(v, a, at, own, Q, c, T);
                    __syncwarp();
                    if (lane < m) to[0] = v[0];
                }
                if (lane < m && up) rows[lane * a.ps + w] = 0u;
                __syncwarp();
            }
        }
    }
    __syncwarp();
    sb_arrive();
    sb_wait();   // the scales are in every CTA, and P is complete; no remote access after this
    if (cta == 0) return;
    // this CTA's columns of P
    for (int i = tid; i < (d + 1) * m * kSbUpd; i += kSbThreads) {
        const int w = ((int)cta - 1) * kSbUpd + (i & (kSbUpd - 1)), tr = i / kSbUpd, t = tr / m, r = tr - t * m;
        if (w < m) a.P[((size_t)t * m + r) * m + w] = red64((u64)rows[r * a.ps + t * m4 + w] * scale[r], a.M);
    }
}
static_assert((kSbCtas - 1) * kSbUpd >= kSbMaxM, "one column of P per warp");

__global__ void k_sb_node(const PmNode n) { pm_node(n, (int)threadIdx.x); }

// Fr = F mod p
__global__ void k_sb_reduce(const u32 *__restrict__ F, long long total, u32 *__restrict__ Fr, const Mod M)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
        Fr[i] = red64(F[i], M);
}

__global__ void k_sb_wiedemann(const u32 *__restrict__ S, long long L, int s, u32 *__restrict__ F, u32 p)
{
    const long long total = L * 2 * s * s;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(i % s);
        const int r = (int)((i / s) % (2 * s));
        const long long k = i / (2LL * s * s);
        u32 v;
        if (r < s) v = S[(k * s + r) * s + j];
        else v = (k == 0 && r - s == j) ? p - 1u : 0u;
        F[i] = v;
    }
}

bool sb_is_prime(u64 q)
{
    // deterministic Miller-Rabin: bases 2, 3, 5, 7 decide every q < 3 215 031 751
    if (q < 2) return false;
    for (u64 sp : {2ull, 3ull, 5ull, 7ull}) {
        if (q == sp) return true;
        if (q % sp == 0) return false;
    }
    u64 dd = q - 1;
    int r = 0;
    while (!(dd & 1)) {
        dd >>= 1;
        ++r;
    }
    auto mulm = [q](u64 x, u64 y) { return (u64)((unsigned __int128)x * y % q); };
    for (u64 b : {2ull, 3ull, 5ull, 7ull}) {
        u64 x = 1, e = dd, base = b % q;
        while (e) {
            if (e & 1) x = mulm(x, base);
            base = mulm(base, base);
            e >>= 1;
        }
        if (x == 1 || x == q - 1) continue;
        bool comp = true;
        for (int i = 1; i < r && comp; ++i) {
            x = mulm(x, x);
            if (x == q - 1) comp = false;
        }
        if (comp) return false;
    }
    return true;
}

size_t sb_round(size_t b) { return (b + kSbAlign - 1) / kSbAlign * kSbAlign; }

// stack bytes of the recursion at order d (degrees at their bound): P1, the
// residual, P2
size_t sb_stack_bytes(int m, int n, long long d, int leaf)
{
    if (d <= leaf) return 0;
    const long long d1 = (d + 1) / 2, d2 = d - d1;
    const size_t mm = (size_t)m * m * 4;
    const size_t P1 = sb_round((d1 + 1) * mm), C = sb_round((size_t)d2 * m * n * 4), P2 = sb_round((d2 + 1) * mm);
    return std::max(P1 + sb_stack_bytes(m, n, d1, leaf), P1 + C + P2 + sb_stack_bytes(m, n, d2, leaf));
}

// nodes (device slots) of the recursion
long long sb_nodes(long long d, int leaf)
{
    if (d <= leaf) return 1;
    return 1 + sb_nodes((d + 1) / 2, leaf) + sb_nodes(d - (d + 1) / 2, leaf);
}

// the largest transform workspace of the recursion: its top products
size_t sb_work_bytes(int m, int n, long long d, long long async)
{
    if (d <= async) return 0;
    const long long d1 = (d + 1) / 2, d2 = d - d1;
    return std::max(pm_product_bytes(m, m, n, d1, d - 1, d1, d - 1), pm_product_bytes(m, m, m, d2, d1, 0, d));
}

struct SbRun {
    u32 p;
    int m, n, base, leaf;   // base: the leaf order of the degree bounds; leaf: orders per M-Basis launch
    long long async;
    Mod M;
    cudaStream_t st;
    char *stack;
    size_t cap, top;
    void *pm_work;
    size_t pm_bytes;
    SbSlot *slots;
    long long nslot, cslot;
};

u32 *sb_alloc(SbRun &R, size_t elems)
{
    const size_t b = sb_round(elems * 4);
    if (R.top + b > R.cap) return nullptr;
    u32 *ptr = reinterpret_cast<u32 *>(R.stack + R.top);
    R.top += b;
    return ptr;
}

template <int N>
ffspmv_status sb_launch(const SbLeaf &a, size_t smem, cudaStream_t st)
{
    // p <= 2^26: all 33 products of a sum stay below p 2^32
    auto *k = a.M.m <= (1u << 26) ? k_sb_mbasis<N, false, false> : k_sb_mbasis<N, true, false>;
    if constexpr (N == 32)
        if (a.M.m == 2u) k = k_sb_mbasis<32, false, true>;
    FF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSbSmemMax));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kSbCtas);
    cfg.blockDim = dim3(kSbThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kSbCtas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    FF_CUDA(cudaLaunchKernelEx(&cfg, k, a));
    return FFSPMV_OK;
}

ffspmv_status sb_leaf(SbRun &R, const u32 *F, long long d, const int *shift, u32 *P, SbSlot *out)
{
    SbLeaf a;
    memset(&a, 0, sizeof(a));
    a.F = F;
    a.P = P;
    a.shift = shift;
    a.out = out;
    a.m = R.m;
    a.n = R.n;
    a.d = (int)d;
    a.rs = sb_rstride(R.n, d);
    a.ps = sb_pstride(R.m, d);
    u32 y = R.p;   // p^-1 mod 2^32 for odd p (Newton)
    for (int i = 0; i < 4; ++i) y *= 2u - R.p * y;
    a.pinv = y;
    a.M = R.M;
    const size_t smem = sb_leaf_smem(R.m, R.n, d);
    if (R.p == 2u) return sb_launch<32>(a, smem, R.st);
    return R.n <= 8 ? sb_launch<8>(a, smem, R.st) : R.n <= 16 ? sb_launch<16>(a, smem, R.st) : sb_launch<32>(a, smem, R.st);
}

// Order-d basis of F (d coefficients of m x n) for the shift at `shift` (device)
// into P ((d+1) coefficients, zero above the degree); its node in *out.
ffspmv_status sb_rec(SbRun &R, const u32 *F, long long d, const int *shift, u32 *P, SbSlot **out)
{
    ffspmv_status st;
    if (R.nslot >= R.cslot) return FFSPMV_ERR_ARG;
    SbSlot *node = *out = R.slots + R.nslot++;
    if (d <= R.leaf) return sb_leaf(R, F, d, shift, P, node);
    const long long d1 = (d + 1) / 2, d2 = d - d1;
    const size_t mm = (size_t)R.m * R.m, mn = (size_t)R.m * R.n;
    const size_t mark = R.top;
    SbSlot *s1 = nullptr, *s2 = nullptr;
    u32 *P1 = sb_alloc(R, (d1 + 1) * mm);
    if (!P1) return FFSPMV_ERR_ARG;
    if ((st = sb_rec(R, F, d1, shift, P1, &s1)) != FFSPMV_OK) return st;
    u32 *C = sb_alloc(R, d2 * mn);   // the residual: coefficients d1..d-1 of P1 F
    u32 *P2 = sb_alloc(R, (d2 + 1) * mm);
    if (!C || !P2) return FFSPMV_ERR_ARG;
    const PmNode pn = {nullptr, nullptr, node, (int)d, d <= R.base ? 1 : 0, R.m};
    if (d <= R.async) {
        st = pm_direct(R.p, R.m, R.m, R.n, (int)d1, (int)d - 1, P1, F, C, (int)d1, (int)d - 1, &s1->e, nullptr, nullptr, R.st);
        if (st != FFSPMV_OK) return st;
        if ((st = sb_rec(R, C, d2, s1->delta, P2, &s2)) != FFSPMV_OK) return st;
        PmNode w = pn;
        w.s1 = s1;
        w.s2 = s2;
        st = pm_direct(R.p, R.m, R.m, R.m, (int)d2, (int)d1, P2, P1, P, 0, (int)d, &s2->e, &s1->e, &w, R.st);
        if (st != FFSPMV_OK) return st;
    } else {
        SbSlot h1, h2;
        FF_CUDA(cudaMemcpyAsync(&h1, s1, sizeof(SbSlot), cudaMemcpyDeviceToHost, R.st));
        FF_CUDA(cudaStreamSynchronize(R.st));
        const long long e1 = h1.e;
        if (e1 < 0 || e1 > d1) return FFSPMV_ERR_CUDA;
        st = pm_product(R.p, R.m, R.m, R.n, e1, d - 1, P1, F, C, d1, d - 1, R.pm_work, R.pm_bytes, R.st);
        if (st != FFSPMV_OK) return st;
        if ((st = sb_rec(R, C, d2, s1->delta, P2, &s2)) != FFSPMV_OK) return st;
        FF_CUDA(cudaMemcpyAsync(&h2, s2, sizeof(SbSlot), cudaMemcpyDeviceToHost, R.st));
        FF_CUDA(cudaStreamSynchronize(R.st));
        const long long e2 = h2.e;
        if (e2 < 0 || e2 > d2) return FFSPMV_ERR_CUDA;
        st = pm_product(R.p, R.m, R.m, R.m, e2, e1, P2, P1, P, 0, e1 + e2, R.pm_work, R.pm_bytes, R.st);
        if (st != FFSPMV_OK) return st;
        if (e1 + e2 < d)
            FF_CUDA(cudaMemsetAsync(P + (e1 + e2 + 1) * mm, 0, (size_t)(d - e1 - e2) * mm * 4, R.st));
        k_sb_node<<<1, 32, 0, R.st>>>(PmNode{s1, s2, node, (int)d, pn.leaf, R.m});
        FF_CUDA(cudaGetLastError());
    }
    R.top = mark;
    return FFSPMV_OK;
}

struct SbLayout {
    int base, leaf;
    long long async, nodes;
    size_t pm, f, slots, stack, total;
};

ffspmv_status sb_layout(int32_t m, int32_t n, int64_t d, int32_t base, SbLayout *out)
{
    if (m < 1 || m > kSbMaxM || n < 1 || n > m || d < 1 || base < 0 || base > kSbMaxBase) return FFSPMV_ERR_ARG;
    SbLayout L;
    L.base = base ? base : kSbMaxBase;
    L.leaf = std::min(L.base, kSbLeaf);
    L.async = kSbAsync;
    if (sb_leaf_smem(m, n, L.leaf) > kSbSmemMax) return FFSPMV_ERR_UNSUPPORTED;
    // the recursion's largest product, ceil(d/2) + d coefficients, must fit the transforms
    if (d > L.base && (d + 1) / 2 + d > (1LL << 15)) return FFSPMV_ERR_UNSUPPORTED;
    L.nodes = sb_nodes(d, L.leaf);
    L.pm = sb_round(sb_work_bytes(m, n, d, L.async));
    L.f = sb_round((size_t)d * m * n * 4);
    L.slots = sb_round(sizeof(SbSlot) * (size_t)(L.nodes + 1));   // and the input shift
    L.stack = sb_stack_bytes(m, n, d, L.leaf);
    L.total = L.pm + L.f + L.slots + L.stack;
    *out = L;
    return FFSPMV_OK;
}

}  // namespace
}  // namespace ff

using namespace ff;

extern "C" ffspmv_status sigma_basis_workspace(int32_t m, int32_t n, int64_t d, int32_t base, int64_t *bytes)
{
    if (!bytes) return FFSPMV_ERR_ARG;
    SbLayout L;
    const ffspmv_status st = sb_layout(m, n, d, base, &L);
    if (st != FFSPMV_OK) return st;
    *bytes = (int64_t)L.total;
    return FFSPMV_OK;
}

extern "C" ffspmv_status sigma_basis(uint32_t p, int32_t m, int32_t n, int64_t d, int32_t base,
                                     const uint32_t *d_F, const int32_t *h_shift, uint32_t *d_P,
                                     int32_t *h_delta, int64_t *h_degree, void *d_work, int64_t work_bytes,
                                     ffspmv_stream_t stream)
{
    if (p < 2 || p > (1u << 31) || !sb_is_prime(p) || !d_F || !d_P || !h_delta || !d_work) return FFSPMV_ERR_ARG;
    SbLayout L;
    ffspmv_status st = sb_layout(m, n, d, base, &L);
    if (st != FFSPMV_OK) return st;
    if (work_bytes < (int64_t)L.total || ((uintptr_t)d_work & 15)) return FFSPMV_ERR_ARG;
    int shift[kSbMaxM] = {};
    if (h_shift) {
        for (int i = 0; i < m; ++i) {
            if (h_shift[i] > kSbMaxShift || h_shift[i] < -kSbMaxShift) return FFSPMV_ERR_ARG;
            shift[i] = h_shift[i];
        }
    }
    SbRun R;
    memset(&R, 0, sizeof(R));
    R.p = p;
    R.m = m;
    R.n = n;
    R.base = L.base;
    R.leaf = L.leaf;
    R.async = L.async;
    R.M = make_mod(p, 1, 0);
    R.st = (cudaStream_t)stream;
    char *w = static_cast<char *>(d_work);
    R.pm_work = w;
    R.pm_bytes = L.pm;
    u32 *Fr = reinterpret_cast<u32 *>(w + L.pm);
    R.slots = reinterpret_cast<SbSlot *>(w + L.pm + L.f);
    R.cslot = L.nodes;
    R.stack = w + L.pm + L.f + L.slots;
    R.cap = L.stack;
    int *d_shift = R.slots[L.nodes].delta;
    FF_CUDA(cudaMemcpyAsync(d_shift, shift, sizeof(shift), cudaMemcpyHostToDevice, R.st));
    const long long total = d * m * n;
    const unsigned blocks = (unsigned)std::min<long long>((total + 255) / 256, 4096);
    k_sb_reduce<<<blocks, 256, 0, R.st>>>(d_F, total, Fr, R.M);
    FF_CUDA(cudaGetLastError());
    SbSlot *root = nullptr, h;
    st = sb_rec(R, Fr, d, d_shift, d_P, &root);
    if (st == FFSPMV_OK) FF_CUDA(cudaMemcpyAsync(&h, root, sizeof(h), cudaMemcpyDeviceToHost, R.st));
    const cudaError_t sync = cudaStreamSynchronize(R.st);
    if (st != FFSPMV_OK) return st;
    FF_CUDA(sync);
    for (int i = 0; i < m; ++i) h_delta[i] = h.delta[i];
    if (h_degree) *h_degree = h.e;
    return FFSPMV_OK;
}

extern "C" ffspmv_status sigma_wiedemann_input(uint32_t p, int32_t s, int64_t L, const uint32_t *d_S, uint32_t *d_F,
                                               ffspmv_stream_t stream)
{
    if (p < 2 || p > (1u << 31) || s < 1 || s > kSbMaxM / 2 || L < 1 || !d_S || !d_F) return FFSPMV_ERR_ARG;
    const long long total = L * 2 * s * s;
    const unsigned blocks = (unsigned)std::min<long long>((total + 255) / 256, 4096);
    k_sb_wiedemann<<<blocks, 256, 0, (cudaStream_t)stream>>>(d_S, L, s, d_F, p);
    FF_CUDA(cudaGetLastError());
    return FFSPMV_OK;
}
