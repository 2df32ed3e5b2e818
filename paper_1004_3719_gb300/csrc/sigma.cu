// Sigma-bases over F_p for the second step of block Wiedemann (Sec. 3.2,
// "Parallelization of the sigma-basis computation"): PM-Basis (Giorgi,
// Jeannerod and Villard, ISSAC 2003) as a host recursion on the order whose
// work is polynomial-matrix products on the GPU (polymat.cu, Sec. 3.2.1's
// evaluation / pointwise / interpolation scheme, and products by definition
// for short operands), and M-Basis, the iterative algorithm Sec. 3.2.2
// recommends at small orders, as one cluster of CTAs per leaf.
//
// The recursion.  An order-d basis is P2 P1 with P1 of order d1 = ceil(d/2)
// and P2 of the residual, the coefficients d1..d-1 of P1 F, with P1's degrees
// as its shift.  M-Basis itself is the recursion's limit (order k's operations
// depend only on that order's residual and the current degrees), so the
// result is the same matrix wherever the leaves are cut; the leaves here take
// at most sb_leaf_max orders.  Up to order kSbAsync a node needs nothing from the
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
// registers.  Panel by panel, its owner shares the panel's columns; every warp
// eliminates these first (the same few operations, redundantly: the chain of
// dependent steps), then applies the steps to its own columns, so that no step
// needs an exchange between warps.  Nearly always the pivots are the rows in
// order, so a panel first takes them as known: a step is then a shuffle and a
// multiply-add long, with no vote on the way; it is done again with votes if
// one of them turns out zero.  The owner's columns turn into the coefficients
// of the pivots, so what comes out is a matrix: every row becomes c r plus a
// combination of the *original* pivot rows.  Eight warps of the first CTA apply
// it to what R_{k+1} needs, and six other CTAs of the cluster, a few columns of
// R and of P each, to all the rest: R's coefficient k + 2 first, which they send
// back for the order after.  So the first CTA does nothing but eliminate, and
// nobody waits for a CTA that falls behind for some orders.
//
// What bounds it: the elimination's chain (about 5 000 clocks per order of a 32
// x 16 leaf: 120 per dependent step, 100 per step to apply, 180 per exchange of
// a panel, 900 for R_{k+1}); the other CTAs take 4 000.  Measured, order
// 12 502, 32 x 16, p = 65521: one cluster of eight CTAs per leaf of order 24-25
// that exchanged every row operation took about 20 us per order and 293 ms for
// the whole basis (with the transforms of polymat.cu); four eliminating warps
// beside eight that apply to R, two CTAs for P, leaves of at most 16 orders, 4.3
// us and 81 ms; R in CTAs of its own 3.5 us and 64 ms; columns of R and P mixed,
// panels before the rest, as it is here, 3.0 us and 58 ms (56 with the products
// of 16-bit pairs, polymat.cu).
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
constexpr long long kSbAsync = 200;         // largest order whose nodes run without the host
constexpr int kSbElim = 4;                  // warps that eliminate (first CTA)
constexpr int kSbRes = 8;                   // warps that bring R's next coefficient up to date (first CTA)
constexpr int kSbWarps = 20;
constexpr int kSbFirst = 32 * (kSbRes + kSbElim);
constexpr int kSbThreads = 32 * kSbWarps;
constexpr int kSbSend = 32 * (kSbWarps - kSbElim);
constexpr int kSbApply = 6;                 // CTAs that apply the operations to P and to R's later coefficients
constexpr int kSbCtas = 1 + kSbApply;
constexpr u32 kSbPolls = 64;                // tries of a wait between two looks at the clock
constexpr u64 kSbWaitNs = 700ull * 1000 * 1000, kSbDrainNs = 50ull * 1000 * 1000;   // its limit; that of messages in flight
constexpr size_t kSbSmemMax = 227 * 1024;
constexpr size_t kSbAlign = 256;
constexpr int kSbMaxShift = 1 << 24;

struct SbLeaf {
    const u32 *F;        // d x m x n residues
    u32 *P;              // out: (d+1) x m x m
    const int *shift;    // m
    SbSlot *out;
    int m, n, d;
    int stride;          // words per row of R and of P in shared memory
    int hold;            // testing: the operations of this order and of the later ones are not sent (else INT_MAX)
    u32 pinv;            // p^-1 mod 2^32 (odd p)
    u32 one;             // 2^32 mod p (p = 2: 1): x -> x under sb_red
    Mod M;
};

// Shared memory of a leaf's CTA: the operations of every order, so that none
// is ever waited for to be read before the next is written; then rows, one of
// the matrix every `stride` words (2 mod 32: the 8-byte pieces that half a warp
// reads of 16 rows lie in distinct banks), a coefficient after the other.  First
// CTA: slot t holds R's coefficient t with the operations of orders 0..t-2
// applied, slots yb and yb + 1 (yb = d, or d + 1 if odd) R_k, all columns (n4 =
// n rounded up to 4).  The
// others: two copies of their columns of R, then of P (an order reads one and
// writes the other).
template <int N>
struct SbOps {
    u32 T[N][kSbMaxM];         // [column][row]: what row gets of the column's pivot row
    u32 c[kSbMaxM];            // [row]: what it keeps of itself
    u32 q[kSbMaxM];            // [column]: byte offset of the pivot row (any row, with T = 0, when there is none)
    u32 isp[kSbMaxM];          // [row]: 1 for the pivot rows
};
typedef u32 SbPanel[2][8][32];   // a panel's columns, by lane of the eliminating warps; two copies
constexpr size_t kSbScaleOff = 0;                                       // the final row scales
constexpr size_t kSbOrdOff = kSbScaleOff + kSbMaxM * 4;                 // [kSbElim][32]
constexpr size_t kSbXOff = kSbOrdOff + kSbElim * 32 * 4;                // SbPanel
constexpr size_t kSbCOff = kSbXOff + sizeof(SbPanel);                   // what rows keep, between panels
constexpr size_t kSbBarOff = kSbCOff + 32 * 4;                         // mbarriers: operations of order k, R's coefficient t
constexpr size_t kSbOpsOff = kSbBarOff + 2 * kSbMaxBase * 8;
static_assert(kSbOpsOff % 16 == 0 && sizeof(SbOps<8>) % 16 == 0, "16-byte pieces");

// The column pairs of R or of P (`cols` columns) that CTA h of kSbApply holds:
// their number and the first.
__host__ __device__ inline int sb_share(int cols, int h, int *first)
{
    const int pairs = (cols + 3) / 4 * 2, q = pairs / kSbApply, r = pairs % kSbApply;
    *first = h * q + (h < r ? h : r);
    return q + (h < r ? 1 : 0);
}

int sb_stride(int m, int n, int d)
{
    int words = (d + 3) * ((n + 3) / 4 * 4), first;
    for (int h = 0; h < kSbApply; ++h)
        words = std::max(words, 4 * d * sb_share(n, h, &first) + 4 * (d + 1) * sb_share(m, kSbApply - 1 - h, &first));
    return (words + 29) / 32 * 32 + 2;
}

size_t sb_leaf_smem(int m, int n, int d, size_t ops) { return kSbOpsOff + d * ops + (size_t)sb_stride(m, n, d) * m * 4; }

// Largest order of one launch: what fits the shared memory, and beyond which
// what the products beside it take is small (order 12 502, 32 x 16: 67 ms at 16,
// 61 at 24, 58 at 32, before the products took 16-bit pairs).
int sb_leaf_max(int n) { return n <= 16 ? 32 : 24; }

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

// The same without the last step, in [0, 2p), where the sums of four such
// products stay below p 2^32 (LAZY: p <= 2^26).  Zero is 0 or p.
template <bool LAZY, bool EVEN>
__device__ __forceinline__ u32 sb_lazy(u64 x, const SbLeaf &a)
{
    if constexpr (LAZY) return (u32)(x >> 32) + a.M.m - __umulhi((u32)x * a.pinv, a.M.m);
    return sb_red<EVEN>(x, a);
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

__device__ __forceinline__ u32 sb_shared(const void *ptr) { return (u32)__cvta_generic_to_shared(ptr); }

// 8 or 16 bytes into another CTA, counted by the mbarrier `bar` there.
__device__ __forceinline__ void sb_send(u32 addr, uint2 v, u32 bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(v.x),
                 "r"(v.y), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void sb_send(u32 addr, uint4 v, u32 bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void sb_bar_init(u32 bar, u32 bytes)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Every mbarrier is used once.  False when the wait ran out: `ns` nanoseconds
// after the first kSbPolls tries (the clock is read every kSbPolls tries; the
// hardware may draw each of them out).
__device__ __forceinline__ bool sb_bar_wait(u32 bar, u64 ns = kSbWaitNs)
{
    u64 t0 = 0;
    for (u32 i = 1;; ++i) {
        u32 ok;
        asm volatile("{\n.reg .pred q;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], 0;\n"
                     "selp.u32 %0, 1, 0, q;\n}"
                     : "=r"(ok)
                     : "r"(bar)
                     : "memory");
        if (ok) return true;
        if (i % kSbPolls) continue;
        const u64 t = global_ns();
        if (t0 == 0) t0 = t;
        else if (t - t0 > ns) return false;
    }
}

__device__ __forceinline__ void sb_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void sb_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// The end of a warp whose wait ran out.  A CTA that gave up at order k sends
// zeros for the coefficients that it owes the first CTA, so that this one ends
// without waiting; and no CTA leaves before what was sent to it has landed.
__device__ __noinline__ void sb_give_up(int *bad, u32 bar, int k0, int k1, u32 to, u32 to_bar, u32 step, int t0)
{
    *bad = 1;
    for (int t = t0; t < k1; ++t) sb_send(to + t * step, make_uint2(0u, 0u), to_bar + 8 * t);
    __syncwarp();
    sb_arrive();
    sb_wait();
    const u64 since = global_ns();
    for (int k = k0; k < k1; ++k) {
        const u64 spent = global_ns() - since;
        sb_bar_wait(bar + 8 * k, spent < kSbDrainNs ? kSbDrainNs - spent : 0);
    }
}

__device__ __forceinline__ u32 sb_rank()
{
    u32 r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// The operations applied to two adjacent columns of one coefficient:
// lane r gets row r's new values.  `row0` points at the columns in row 0.
// FOLD (p > 2^26): two products below p^2 are added to a sum below p 2^32,
// then the sum is brought back below that; else all 33 fit.
__device__ __forceinline__ uint2 sb_at(const u32 *row0, u32 bytes)
{
    return *reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(row0) + bytes);
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
template <int N, bool FOLD, bool EVEN>
__device__ __forceinline__ uint2 sb_apply(const SbLeaf &a, const u32 *row0, u32 own_off, const SbPiv<N> &Q, u32 c, const u32 (&T)[N])
{
    const u32 p = a.M.m;
    const uint2 own = sb_at(row0, own_off);
    u64 x = (u64)c * own.x, y = (u64)c * own.y;
#pragma unroll
    for (int j = 0; j < N; j += 2) {
        const uint2 v0 = sb_at(row0, Q.at(j)), v1 = sb_at(row0, Q.at(j + 1));
        x += (u64)T[j] * v0.x;
        y += (u64)T[j] * v0.y;
        x += (u64)T[j + 1] * v1.x;
        y += (u64)T[j + 1] * v1.y;
        if (FOLD) {
            x = sb_fold(x, p);
            y = sb_fold(y, p);
        }
    }
    return make_uint2(sb_red<EVEN>(x, a), sb_red<EVEN>(y, a));
}

// N: 8, 16 or 32, at least n.  One cluster of kSbCtas CTAs: the first
// eliminates, the others hold P and R's later coefficients, a few columns each.
// All that moves between them is counted by mbarriers, each used once, in the
// CTA that waits for it: the operations of an order (to all the others), and a
// coefficient of R (to the first) one order before it is needed.
template <int N, bool FOLD, bool EVEN>
__global__ void __launch_bounds__(kSbThreads, 1) k_sb_mbasis(const __grid_constant__ SbLeaf a)
{
    extern __shared__ __align__(16) unsigned char sb_sm[];
    const int m = a.m, n = a.n, d = a.d, S = a.stride;
    const u32 p = a.M.m;
    const int n4 = (n + 3) & ~3, yb = d + (d & 1);
    SbOps<N> *ops = reinterpret_cast<SbOps<N> *>(sb_sm + kSbOpsOff);
    u32 *scale = reinterpret_cast<u32 *>(sb_sm + kSbScaleOff);
    u32 *rows = reinterpret_cast<u32 *>(ops + d);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const u32 cta = sb_rank();
    const u32 bar_ops = sb_shared(sb_sm + kSbBarOff), bar_R = bar_ops + 8 * kSbMaxBase;
    // this CTA's columns: those of R, then those of P (where R's are more, fewer)
    const int h = cta ? (int)cta - 1 : 0;
    int r_first, p_first;
    const int rp = sb_share(n, h, &r_first), pp = sb_share(m, kSbApply - 1 - h, &p_first);
    u32 *P0 = rows + 4 * d * rp;   // (the two copies of R before it)

    if (tid < d) {
        if (cta) sb_bar_init(bar_ops + 8 * tid, (u32)sizeof(SbOps<N>));
        else sb_bar_init(bar_R + 8 * tid, (u32)(m * n4 * 4));
    }
    if (cta == 0 && tid == 0) a.out->bad = 0;
    __syncwarp();
    sb_arrive();
    if (cta == 0) {
        // R's coefficients 0 (as R_0) and 1
        for (int i = tid; i < min(d, 2) * m * n4; i += kSbThreads) {
            const int c = i % n4, tr = i / n4, t = tr / m, r = tr - t * m;
            rows[r * S + (t ? 1 : yb) * n4 + c] = c < n ? __ldg(a.F + ((size_t)t * m + r) * n + c) : 0u;
        }
    } else if (lane < m) {
        for (int t = 1 + warp; t < d; t += kSbWarps)
            for (int c = 0; c < 2 * rp; ++c)
                rows[lane * S + t * 2 * rp + c] =
                    2 * r_first + c < n ? __ldg(a.F + ((size_t)t * m + lane) * n + 2 * r_first + c) : 0u;
        if (warp < 2 * pp) P0[lane * S + warp] = 2 * p_first + warp == lane ? 1u : 0u;   // P = identity
    }
    __syncthreads();
    sb_wait();   // every CTA's mbarriers are ready
    bool ok = true;
    int kf = 0;   // the order at which this CTA gave up

    if (cta == 0 && warp >= kSbWarps - kSbElim) {
        // the eliminating warps: each keeps row r's degree and scale in lane r
        constexpr int NC = N / kSbElim;   // columns per warp: ew NC ...
        const int ew = warp - (kSbWarps - kSbElim), col0 = ew * NC;
        int *ord = reinterpret_cast<int *>(sb_sm + kSbOrdOff) + ew * 32;
        auto &X = *reinterpret_cast<SbPanel *>(sb_sm + kSbXOff);
        u32 *xc = reinterpret_cast<u32 *>(sb_sm + kSbCOff);
        constexpr bool LAZY = !FOLD && !EVEN;
        const int last = (n - 1) / NC;    // the last panel; its warp ends with c and keeps the scales
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
            const u32 *src = rows + (live ? row : 0) * S + (yb + (k & 1)) * n4 + col0;
#pragma unroll
            for (int s = 0; s < NC; ++s) R[s] = live && col0 + s < n ? src[s] : 0u;
            u32 c = 1u;
            bool isp = false;
            int q_of = 31;   // lane j: lane of column j's pivot row (31: the first row, for columns without one)
#pragma unroll 1
            for (int w = 0; w <= last; ++w) {
                const bool mine = ew == w;
                u32 *xs = &X[w & 1][0][0];
                if (mine) {
#pragma unroll
                    for (int j = 0; j < NC; ++j) xs[j * 32 + lane] = R[j];
                }
                if (ew == w - 1) xc[lane] = c;
                asm volatile("bar.sync 3, %0;" ::"n"(kSbElim * 32) : "memory");
                u32 pc[NC];   // the panel's columns
#pragma unroll
                for (int j = 0; j < NC; ++j) pc[j] = xs[j * 32 + lane];
                if (mine && w) c = xc[lane];
                // Step j with pivot lane q[j]: row <- av row - x pivot row
                // (times 2^-32) for some rows, the others as they are: row <-
                // A row + G pivot row.  The panel's own columns first, in which
                // the pivots are found; everything else follows.
                u32 A[NC], G[NC];
                int q[NC];
                auto step = [&](int j, bool act, u32 av) {
                    A[j] = act ? av : a.one;
                    G[j] = act ? (LAZY ? 2 * p : p) - pc[j] : 0u;
#pragma unroll
                    for (int i = 0; i < NC; ++i)
                        if (i > j)
                            pc[i] = sb_lazy<LAZY, EVEN>((u64)G[j] * __shfl_sync(0xffffffffu, pc[i], q[j]) + (u64)A[j] * pc[i], a);
                };
                // first with the rows in order as pivots, lanes 31 - w NC,
                // 30 - w NC ..: right if the panels before took the lanes
                // above and no pivot is zero
                const u32 above = w == 0 ? 0u : ~0u << (32 - NC * w);
                bool good = w * NC + NC <= n && __ballot_sync(0xffffffffu, isp) == above;
                if (good) {
                    bool zero = false;
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        q[j] = 31 - w * NC - j;
                        const u32 av = __shfl_sync(0xffffffffu, pc[j], q[j]);
                        zero = zero || av == 0u || (LAZY && av == p);
                        step(j, lane < q[j], av);
                    }
                    good = !zero;
                    if (good) {
                        isp = lane >= 32 - w * NC - NC;
                        if (lane >= w * NC && lane < w * NC + NC) q_of = 31 - lane;
                    }
                }
                if (!good) {
#pragma unroll
                    for (int j = 0; j < NC; ++j) pc[j] = xs[j * 32 + lane];
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        const bool cand = !isp && pc[j] != 0u && !(LAZY && pc[j] == p);
                        const u32 b = __ballot_sync(0xffffffffu, cand);
                        // (no candidate: the column is zero in every row left,
                        // nothing is taken over and the coefficients are 0)
                        q[j] = b ? 31 - __clz(b) : 31;
                        step(j, cand && lane != q[j], __shfl_sync(0xffffffffu, pc[j], q[j]));
                        isp = isp || (cand && lane == q[j]);
                        if (lane == w * NC + j) q_of = q[j];
                    }
                }
                // the other columns; the owner's turn into the coefficients of
                // the pivots, one with each step
                if (mine) {
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        const u32 cq = __shfl_sync(0xffffffffu, c, q[j]);
#pragma unroll
                        for (int i = 0; i < j; ++i)
                            R[i] = sb_lazy<LAZY, EVEN>((u64)G[j] * __shfl_sync(0xffffffffu, R[i], q[j]) + (u64)A[j] * R[i], a);
                        R[j] = sb_lazy<LAZY, EVEN>((u64)G[j] * cq, a);
                        c = sb_lazy<LAZY, EVEN>((u64)A[j] * c, a);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < NC; ++j)
#pragma unroll
                        for (int i = 0; i < NC; ++i)
                            R[i] = sb_lazy<LAZY, EVEN>((u64)G[j] * __shfl_sync(0xffffffffu, R[i], q[j]) + (u64)A[j] * R[i], a);
                }
            }
            if (LAZY) {
#pragma unroll
                for (int s = 0; s < NC; ++s) R[s] = min(R[s], R[s] - p);
                c = min(c, c - p);
            }
            SbOps<N> &O = ops[k];
            const int qrow = ord[q_of];   // always a row below m: candidates are, and so is the first in the order
            const u32 pb = __ballot_sync(0xffffffffu, isp);
            // rows past m too: zeros
#pragma unroll
            for (int s = 0; s < NC; ++s) O.T[col0 + s][row] = R[s];
            if (ew == last) O.c[row] = c;
            if (ew == 1) O.isp[row] = isp ? 1u : 0u;
            if (ew == 2) O.q[lane] = (u32)(qrow * S * 4);
            // the operations of order k are complete: the other warps go on
            // (this one meets them again when it has to have R)
            asm volatile("bar.arrive 2, %0;" ::"n"(kSbThreads) : "memory");
            const u32 cr = __shfl_sync(0xffffffffu, c, rank);
            if (lane < m) {
                dl += (int)((pb >> rank) & 1u);
                tot = sb_red<EVEN>((u64)tot * cr, a);
            }
        }
        if (ew == last) {
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
        // R_{k+1} is there (which is urgent, and as busy with shared memory)
        constexpr int kPieces = (int)(sizeof(SbOps<N>) / 16), kSend = kSbSend - 32 * kSbRes;
        for (int k = 0; k < d; ++k) {
            asm volatile("bar.sync 2, %0;" ::"n"(kSbThreads) : "memory");
            asm volatile("bar.sync 4, %0;" ::"n"(kSbSend) : "memory");
            const uint4 *src = reinterpret_cast<const uint4 *>(ops + k);
            if (k >= a.hold) continue;
            for (int i = tid - 32 * kSbRes; i < kPieces * (kSbCtas - 1); i += kSend) {
                const u32 r = 1 + i / kPieces, e = i % kPieces;
                sb_send(sb_remote(src + e, r), src[e], sb_remote(sb_sm + kSbBarOff + 8 * k, r));
            }
        }
    } else if (cta == 0) {
        // R_{k+1} from R_k (the pivot rows, which move up by one coefficient)
        // and from coefficient k + 1 (the others)
        const u32 own = (u32)(min(lane, m - 1) * S * 4);
        for (int k = 0; k < d; ++k) {
            if (k && k + 1 < d) ok = __all_sync(0xffffffffu, ok && sb_bar_wait(bar_R + 8 * (k + 1)));
            asm volatile("bar.sync 2, %0;" ::"n"(kSbThreads) : "memory");
            if (k + 1 == d) {
                asm volatile("bar.arrive 4, %0;" ::"n"(kSbSend) : "memory");
                break;
            }
            const SbOps<N> &O = ops[k];
            const u32 c = O.c[lane];
            const u32 *at = rows + (O.isp[lane] ? yb + (k & 1) : k + 1) * n4;
            u32 T[N];
#pragma unroll
            for (int j = 0; j < N; ++j) T[j] = O.T[j][lane];
            const SbPiv<N> Q(O.q);
            for (int u = 2 * warp; u < n4; u += 2 * kSbRes) {
                const uint2 v = sb_apply<N, FOLD, EVEN>(a, at + u, own, Q, c, T);
                if (lane < m) *reinterpret_cast<uint2 *>(rows + lane * S + (yb + ((k + 1) & 1)) * n4 + u) = v;
            }
            asm volatile("bar.arrive 1, %0;" ::"n"(kSbFirst) : "memory");
            asm volatile("bar.arrive 4, %0;" ::"n"(kSbSend) : "memory");
        }
    } else {
        // The operations of order k applied to this CTA's columns, a column
        // pair of a coefficient per warp and turn: of R from coefficient k + 1
        // on, the new k + 2 first, for which the first CTA waits; of P up to k.
        const u32 own = (u32)(min(lane, m - 1) * S * 4);
        const u32 rdiv = rp ? (65536u + rp - 1) / rp : 0u, pdiv = pp ? (65536u + pp - 1) / pp : 0u;   // u / rp: u rdiv >> 16
        for (int k = 0; k < d; ++k) {
            // without the operations nothing is done (their offsets are not there)
            ok = __all_sync(0xffffffffu, sb_bar_wait(bar_ops + 8 * k));
            ok = __syncthreads_and(ok) != 0;
            if (!ok) {
                kf = k;
                break;
            }
            const SbOps<N> &O = ops[k];
            const u32 c = O.c[lane];
            const int up = O.isp[lane] ? 1 : 0;   // pivot rows move up by one coefficient
            u32 T[N];
#pragma unroll
            for (int j = 0; j < N; ++j) T[j] = O.T[j][lane];
            const SbPiv<N> Q(O.q);
            const u32 *Rf = rows + (k & 1) * (2 * d * rp), *Pf = P0 + (k & 1) * (2 * (d + 1) * pp);
            u32 *Rt = rows + ((k + 1) & 1) * (2 * d * rp) + lane * S, *Pt = P0 + ((k + 1) & 1) * (2 * (d + 1) * pp) + lane * S;
            const int nr = k + 2 < d ? (d - 2 - k) * rp : 0, nu = nr + (k + 1) * pp, urgent = nr ? rp : 0;
            if (warp < urgent) {
                const uint2 v = sb_apply<N, FOLD, EVEN>(a, Rf + ((k + 2 - up) * rp + warp) * 2, own, Q, c, T);
                if (lane < m) {
                    *reinterpret_cast<uint2 *>(Rt + ((k + 2) * rp + warp) * 2) = v;
                    sb_send(sb_remote(rows + lane * S + (k + 2) * n4 + 2 * (r_first + warp), 0), v,
                            sb_remote(sb_sm + kSbBarOff + 8 * (kSbMaxBase + k + 2), 0));
                }
            }
            for (int u = warp < urgent ? warp + kSbWarps - urgent : warp - urgent; u < nu; u += kSbWarps) {
                const bool is_R = u < nr;
                const int e = is_R ? u : u - nr, t0 = (int)((u32)e * (is_R ? rdiv : pdiv) >> 16), pr = e - t0 * (is_R ? rp : pp);
                const int t = is_R ? k + 2 + t0 : t0, step = 2 * (is_R ? rp : pp);
                const uint2 v = sb_apply<N, FOLD, EVEN>(a, (is_R ? Rf : Pf) + t * step + 2 * pr, own, Q, c, T);
                u32 *to = (is_R ? Rt : Pt) + 2 * pr;
                if (lane < m) {
                    const uint2 zero = make_uint2(0u, 0u);
                    if (!is_R || (t + up < d && t + up > k + 2)) *reinterpret_cast<uint2 *>(to + (t + up) * step) = v;
                    // P: what no coefficient moves to
                    if (!is_R && t == 0 && up) *reinterpret_cast<uint2 *>(to) = zero;
                    if (!is_R && t == k && !up) *reinterpret_cast<uint2 *>(to + (k + 1) * step) = zero;
                }
            }
        }
    }
    if (!ok) {
        const bool owes = cta && warp < rp && lane < m;
        sb_give_up(&a.out->bad, cta ? bar_ops : bar_R, cta ? 0 : 2, d, sb_remote(rows + lane * S + 2 * (r_first + warp), 0),
                   sb_remote(sb_sm + kSbBarOff + 8 * kSbMaxBase, 0), 4 * n4, owes ? kf + 2 : d);
    } else {
        __syncwarp();
        sb_arrive();
        sb_wait();   // the scales are in every CTA; no remote access is begun after this
    }
    if (cta == 0 || lane >= m) return;
    // this CTA's columns of P
    const u32 *Pd = P0 + (d & 1) * (2 * (d + 1) * pp) + lane * S;
    const u32 sc = scale[lane];
    for (int t = warp; t <= d; t += kSbWarps)
        for (int c = 0; c < 2 * pp; ++c)
            if (2 * p_first + c < m) a.P[((size_t)t * m + lane) * m + 2 * p_first + c] = red64((u64)Pd[t * 2 * pp + c] * sc, a.M);
}
static_assert(kSbMaxM / 2 <= kSbWarps * kSbApply, "a warp per column pair of R's next coefficient");
static_assert(2 * ((kSbMaxM / 2 + kSbApply - 1) / kSbApply) <= kSbWarps, "a warp per column of P's first coefficient");

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
    int hold;
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
ffspmv_status sb_launch(const SbLeaf &a, cudaStream_t st)
{
    const size_t smem = sb_leaf_smem(a.m, a.n, a.d, sizeof(SbOps<N>));
    // p <= 2^26: all 33 products of a sum stay below p 2^32
    auto *k = a.M.m <= (1u << 26) ? k_sb_mbasis<N, false, false> : k_sb_mbasis<N, true, false>;
    if (a.M.m == 2u) k = k_sb_mbasis<N, false, true>;
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
    a.stride = sb_stride(R.m, R.n, a.d);
    a.hold = R.hold;
    R.hold = INT_MAX;   // (the first leaf's only)
    u32 y = R.p;   // p^-1 mod 2^32 for odd p (Newton)
    for (int i = 0; i < 4; ++i) y *= 2u - R.p * y;
    a.pinv = y;
    a.one = R.p == 2u ? 1u : (u32)((1ull << 32) % R.p);
    a.M = R.M;
    return R.n <= 8 ? sb_launch<8>(a, R.st) : R.n <= 16 ? sb_launch<16>(a, R.st) : sb_launch<32>(a, R.st);
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
        if (h1.bad) return FFSPMV_ERR_TIMEOUT;
        const long long e1 = h1.e;
        if (e1 < 0 || e1 > d1) return FFSPMV_ERR_CUDA;
        st = pm_product(R.p, R.m, R.m, R.n, e1, d - 1, P1, F, C, d1, d - 1, R.pm_work, R.pm_bytes, R.st);
        if (st != FFSPMV_OK) return st;
        if ((st = sb_rec(R, C, d2, s1->delta, P2, &s2)) != FFSPMV_OK) return st;
        FF_CUDA(cudaMemcpyAsync(&h2, s2, sizeof(SbSlot), cudaMemcpyDeviceToHost, R.st));
        FF_CUDA(cudaStreamSynchronize(R.st));
        if (h2.bad) return FFSPMV_ERR_TIMEOUT;
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
    L.leaf = std::min(L.base, sb_leaf_max(n));
    L.async = kSbAsync;
    if (sb_leaf_smem(m, n, L.leaf, n <= 16 ? sizeof(SbOps<16>) : sizeof(SbOps<32>)) > kSbSmemMax) return FFSPMV_ERR_UNSUPPORTED;
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

static ffspmv_status sb_basis(uint32_t p, int32_t m, int32_t n, int64_t d, int32_t base, const uint32_t *d_F,
                              const int32_t *h_shift, uint32_t *d_P, int32_t *h_delta, int64_t *h_degree, void *d_work,
                              int64_t work_bytes, int hold, ffspmv_stream_t stream)
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
    R.hold = hold;
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
    if (h.bad) return FFSPMV_ERR_TIMEOUT;
    for (int i = 0; i < m; ++i) h_delta[i] = h.delta[i];
    if (h_degree) *h_degree = h.e;
    return FFSPMV_OK;
}

extern "C" ffspmv_status sigma_basis(uint32_t p, int32_t m, int32_t n, int64_t d, int32_t base,
                                     const uint32_t *d_F, const int32_t *h_shift, uint32_t *d_P,
                                     int32_t *h_delta, int64_t *h_degree, void *d_work, int64_t work_bytes,
                                     ffspmv_stream_t stream)
{
    return sb_basis(p, m, n, d, base, d_F, h_shift, d_P, h_delta, h_degree, d_work, work_bytes, INT_MAX, stream);
}

extern "C" ffspmv_status ffspmv_sigma_basis_hold(uint32_t p, int32_t m, int32_t n, int64_t d, int32_t base,
                                                 const uint32_t *d_F, const int32_t *h_shift, uint32_t *d_P,
                                                 int32_t *h_delta, int64_t *h_degree, void *d_work, int64_t work_bytes,
                                                 int32_t hold, ffspmv_stream_t stream)
{
    if (hold < 0) return FFSPMV_ERR_ARG;
    return sb_basis(p, m, n, d, base, d_F, h_shift, d_P, h_delta, h_degree, d_work, work_bytes, hold, stream);
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
