// The block Wiedemann matrix sequence S_i = X^T A^i Y (mod p), Sec. 3 step 1,
// kept on the device as Sec. 2.5.2 asks.
//
// Persistent path (p <= 2^16, s <= 16, A square, at most 16 entries per row
// once a few dense diagonals are merged): one cooperative kernel runs every
// step.  CTA c owns a contiguous slice of rows, its warps 16-row groups: two
// lanes per row gather the 16-residue rows of V_i that the row's entries name
// (32 bytes each, from L2), form the row of V_{i+1}, store it, and the warp
// projects its 16 rows on the matching rows of X with tensor-core MMAs on
// 8-bit limbs, without meeting the other warps.  A bounded grid barrier then
// publishes V_{i+1}; each CTA sums and writes its partial projection after it
// has arrived there, and a warp of its own adds the CTAs' partials of a step up
// during the step after next.  The kernel is captured in a CUDA graph.
//
// Per-launch path (everything else): for every step one projection launch and
// the plan's SpMM launches.
//
// Arithmetic.  Two entries' residues of one component in a 32-bit word and the
// two values as four bytes: two dp2a instructions (16 x 8 bits, two products
// each) do two multiply-adds, the low and the high bytes of the values in
// sums of their own (at most 16 products below 2^24 each), at half the
// multiplier's time of 64-bit multiply-adds; the two sums are joined and
// reduced in 32 bits.
//
// Exactness of the projection on tensor cores: a residue v < 2^16 splits as
// v = 256*h + l with h, l < 256, both exact in fp16; a 16-row group adds
// below 2^20 to an fp32 accumulator of limb products (twice that where the
// two cross terms share one), which stays an exact integer below 2^23 over
// kSeqTiles groups and is then folded into integers mod p.
//
// Measured, 100 000 x 100 000, 9.5 entries per row, s = 16, p = 65521: 15.1 us
// per step with 64-bit multiply-adds, row passes that met at CTA barriers and
// projections published before the barrier; 7.55 us with warps of their own
// and dp2a, 7.1 us with the projection after the arrival.  Of a step's 13.9
// thousand clocks the gathers take about 10: 0.95 million 32-byte rows from
// L2, one line each, near the rate at which this chip serves random sectors
// (about 250 G/s).
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "ff_block.h"
#include "ff_internal.cuh"
#include "ff_select.h"

namespace ff {

namespace {

constexpr int kSeqWorkers = 15;                   // warps that multiply (19: 94.7 ms for 12 502 steps, 23: 91.2, 15: 89.0)
constexpr int kSeqWarps = kSeqWorkers + 1;        // ... and the one that sums the CTAs' partial projections
constexpr int kSeqThreads = 32 * kSeqWarps;
constexpr int kS = 16;                            // block width of the persistent kernel
constexpr int kMaxEnt = 16;                       // entries per row
constexpr int kSeqBatch = 5;                      // entry pairs gathered together per lane
constexpr int kSeqTiles = 3;                      // groups that a warp forms before it projects them
constexpr int kSeqBufs = 3;                       // partial projections in flight
constexpr long long kSeqBuildSteps = 48;          // steps for which a block layout is built (p > 2^16)
constexpr int kVsStride = 24;                     // halves per staged row (no bank conflicts for ldmatrix)
constexpr unsigned kDefaultSpins = 1u << 22;      // x <= 64 ns sleeps: well under a second

struct SeqArgs {
    long long n;
    int s;
    int npair;                 // entry pairs per row
    long long ld;
    long long nsteps;
    const u32 *col;            // [2 npair][ld]: columns (value 0: the row itself)
    const u32 *val;            // [npair][ld]: bytes (v0 low, v1 low, v0 high, v1 high)
    const unsigned char *gnp;  // [n / 16]: pairs in use in a 16-row group
    const uint4 *XF;           // X limbs in MMA A-fragment order: [n/16][limb][lane]
    unsigned short *V0, *V1;   // n x 16
    u32 *partial;              // [kSeqBufs][nblocks][256]
    u32 *S;
    u32 *Vnext;
    unsigned *bar;             // [0] arrivals
    int *status;               // [0] timeout flag
    unsigned spin_limit;
    int test_skip;
    int xf_smem;               // X fragments of the CTA's rows held in shared memory
    int mat_smem;              // the CTA's rows of the matrix held in shared memory
    int mrows;                 // rows of one CTA's resident matrix slice (capacity)
    int mat_off;               // byte offset of that slice in dynamic shared memory
    Mod M;
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int ld_volatile_int(const int *p)
{
    int v;
    asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier with a bounded wait, in two halves.  The arrival counter
// (zeroed before the launch) only grows: barrier number `epoch` is passed once
// it reaches epoch * gridDim.x.  One thread per CTA adds its arrival with
// release order (after the CTA's __syncthreads, so it publishes the whole
// CTA's writes) and polls with acquire loads.  The wait returns false (and
// sets status[0]) when it ran out or another CTA already gave up.
__device__ __forceinline__ void grid_arrive(const SeqArgs &a, bool skip)
{
    __syncthreads();
    if (threadIdx.x == 0 && !skip) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
}

__device__ bool grid_wait(const SeqArgs &a, bool skip, unsigned epoch)
{
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        int ok = 1;
        unsigned it = 0;
        if (!skip) {
            const unsigned target = epoch * gridDim.x;
            while ((int)(ld_acquire(a.bar) - target) < 0) {
                if (++it > a.spin_limit || ((it & 255u) == 0 && ld_volatile_int(a.status) != 0)) {
                    atomicExch(a.status, 1);
                    ok = 0;
                    break;
                }
                if (it > 64) __nanosleep(32);
            }
        } else {
            // test hook: never arrived; wait (bounded) for the others to give up
            while (ld_volatile_int(a.status) == 0 && ++it <= a.spin_limit) __nanosleep(64);
            atomicExch(a.status, 1);
            ok = 0;
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Two 8-bit integers (bits 0-7 and 16-23 of p) as an exact f16x2 pair:
// 0x6400 | b is the half 1024 + b, and subtracting 1024 is exact.
__device__ __forceinline__ u32 bytes_to_half2(u32 p)
{
    u32 r;
    asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(p | 0x64006400u), "r"(0x64006400u));
    return r;
}

// An exact non-negative integer below 2^23 held in an fp32, as u32.
__device__ __forceinline__ u32 f32_to_u32(float f)
{
    return __float_as_uint(f + 8388608.0f) - 0x4B000000u;
}

__device__ __forceinline__ void mma16816(float (&d)[4], const uint4 &A, u32 b0, u32 b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(A.x), "r"(A.y), "r"(A.z), "r"(A.w), "r"(b0), "r"(b1));
}

struct __align__(16) SeqSmem {
    u32 red[kSeqWorkers][kS * kS];                       // per-warp partial projections
    unsigned short vs[kSeqWorkers][kSeqTiles][16 * kVsStride];  // per-warp staged rows of V
};
constexpr size_t kXfSmemMax = 225 * 1024 - sizeof(SeqSmem);  // shared memory for resident X fragments and matrix rows

// t mod m up to m (in [0, 2m)), mu = floor(2^32 / m) (Barrett, 1986)
__device__ __forceinline__ u32 seq_mod2(u32 t, u32 m, u32 mu) { return t - __umulhi(t, mu) * m; }
// lo + 256 hi mod m for lo, hi < 2^29
__device__ __forceinline__ u32 seq_join(u32 lo, u32 hi, u32 m, u32 mu)
{
    const u32 t = seq_mod2(seq_mod2(hi, m, mu) * 256u + lo, m, mu);   // hi mod m < 2^17, the sum below 2^30
    return min(t, t - m);
}

// One warp's fp32 sums of limb products: rows 8h + g of X^T against columns
// 8 nt + 2t, 2t + 1: [weight 1, 256, 65536][nt][e].
struct SeqSums {
    float d[3][2][4];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int w = 0; w < 3; ++w)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) d[w][nt][e] = 0.0f;
    }
};

// The sums, mod p, into (first) or onto this warp's words of sm.red.
__device__ __forceinline__ void seq_flush(const SeqArgs &a, u32 *red, SeqSums &P, bool first, u32 mu)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const u32 cross = f32_to_u32(P.d[1][nt][e]), hi = f32_to_u32(P.d[2][nt][e]), lo = f32_to_u32(P.d[0][nt][e]);
            const u32 v = seq_join(lo, seq_join(cross, hi, a.M.m, mu), a.M.m, mu);
            u32 *r = red + (g + (e >> 1) * 8) * kS + nt * 8 + 2 * t + (e & 1);
            *r = first ? v : *r + v;
        }
}

// X^T times the staged rows of a worker warp's groups base, base +
// kSeqWorkers, ... (at most kSeqTiles of them) into (first) or onto its words
// of sm.red.
__device__ __forceinline__ void seq_project(const SeqArgs &a, SeqSmem &sm, const uint4 *xf, int base, int ngroups, bool first,
                                            u32 mu)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncwarp();   // the rows are staged
    SeqSums P;
    P.zero();
    for (int k = 0; k < kSeqTiles; ++k) {
        const int grp = base + k * kSeqWorkers;
        if (grp >= ngroups) break;
        // B fragments of both column tiles: rows 0-7 and 8-15 of each
        u32 b[4];
        const u32 at = (u32)__cvta_generic_to_shared(
            sm.vs[w][k] + ((lane & 7) + ((lane >> 3) & 1) * 8) * kVsStride + (lane >> 4) * 8);
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                     : "r"(at)
                     : "memory");
        const uint4 *f = xf + (size_t)grp * 64 + lane;
        const uint4 A0 = f[0], A1 = f[32];
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const u32 b0 = b[2 * nt], b1 = b[2 * nt + 1];
            const u32 l0 = bytes_to_half2(b0 & 0x00ff00ffu), l1 = bytes_to_half2(b1 & 0x00ff00ffu);
            const u32 h0 = bytes_to_half2((b0 >> 8) & 0x00ff00ffu), h1 = bytes_to_half2((b1 >> 8) & 0x00ff00ffu);
            mma16816(P.d[0][nt], A0, l0, l1);
            mma16816(P.d[1][nt], A0, h0, h1);
            mma16816(P.d[1][nt], A1, l0, l1);
            mma16816(P.d[2][nt], A1, h0, h1);
        }
    }
    seq_flush(a, sm.red[w], P, first, mu);
    __syncwarp();   // the fragments have been read
}

// A worker warp's 16-row groups of rows [r0, r1): V_out = A V_in (when
// COMPUTE; else V_in itself), staged for the projection kSeqTiles groups at a
// time.  All but the last of these batches are projected here (their sums need
// the registers that the gathers take); the first group of the last one is
// returned for seq_project, which then runs after the CTA has arrived at the
// grid barrier.  `col`, `val`, `gnp` start at row r0 with `ld` rows per entry.
template <bool COMPUTE>
__device__ __forceinline__ int seq_rows(const SeqArgs &a, SeqSmem &sm, const uint4 *xf, const u32 *col, const u32 *val,
                                         const unsigned char *gnp, size_t ld, const unsigned short *Vin,
                                         unsigned short *Vout, int r0, int r1, bool project, u32 mu)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int c0 = (lane & 1) * 8;
    const int ngroups = (r1 - r0 + 15) >> 4;
    for (int base = w;; base += kSeqTiles * kSeqWorkers) {
        for (int k = 0; k < kSeqTiles; ++k) {
            const int grp = base + k * kSeqWorkers;
            if (grp >= ngroups) break;
            const int lr = grp * 16 + (lane >> 1), row = r0 + lr;
            uint4 out = make_uint4(0u, 0u, 0u, 0u);
            if (COMPUTE) {
                u32 lo[8], hi[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) lo[i] = hi[i] = 0u;
                const int np = gnp[grp];   // warp-uniform
                const bool live = row < r1;
                const u32 *cp = col + lr, *vp = val + lr;
                const unsigned short *vin = Vin + c0;
                for (int p0 = 0; p0 < np; p0 += kSeqBatch) {
                    uint4 q[kSeqBatch][2];
                    u32 v[kSeqBatch];
#pragma unroll
                    for (int u = 0; u < kSeqBatch; ++u) {
                        q[u][0] = q[u][1] = make_uint4(0u, 0u, 0u, 0u);
                        v[u] = 0u;
                        if (p0 + u < np && live) {
                            const u32 j0 = cp[(size_t)(2 * (p0 + u)) * ld], j1 = cp[(size_t)(2 * (p0 + u) + 1) * ld];
                            v[u] = vp[(size_t)(p0 + u) * ld];
                            q[u][0] = __ldcg(reinterpret_cast<const uint4 *>(vin + (size_t)j0 * kS));
                            q[u][1] = __ldcg(reinterpret_cast<const uint4 *>(vin + (size_t)j1 * kS));
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kSeqBatch; ++u) {
                        const u32 x0[4] = {q[u][0].x, q[u][0].y, q[u][0].z, q[u][0].w};
                        const u32 x1[4] = {q[u][1].x, q[u][1].y, q[u][1].z, q[u][1].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const u32 e0 = __byte_perm(x0[i], x1[i], 0x5410), e1 = __byte_perm(x0[i], x1[i], 0x7632);
                            lo[2 * i] = __dp2a_lo(e0, v[u], lo[2 * i]);
                            hi[2 * i] = __dp2a_hi(e0, v[u], hi[2 * i]);
                            lo[2 * i + 1] = __dp2a_lo(e1, v[u], lo[2 * i + 1]);
                            hi[2 * i + 1] = __dp2a_hi(e1, v[u], hi[2 * i + 1]);
                        }
                    }
                }
                u32 r[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) r[i] = seq_join(lo[i], hi[i], a.M.m, mu);
                out = make_uint4(r[0] | r[1] << 16, r[2] | r[3] << 16, r[4] | r[5] << 16, r[6] | r[7] << 16);
                if (live) *reinterpret_cast<uint4 *>(Vout + (size_t)row * kS + c0) = out;
            } else if (row < r1) {
                out = __ldcg(reinterpret_cast<const uint4 *>(Vin + (size_t)row * kS + c0));
            }
            *reinterpret_cast<uint4 *>(sm.vs[w][k] + (lane >> 1) * kVsStride + c0) = out;
        }
        if (base + kSeqTiles * kSeqWorkers >= ngroups) return base;
        if (project) seq_project(a, sm, xf, base, ngroups, base == w, mu);
    }
}
// both cross products of kSeqTiles groups of 16 rows stay below 2^23 (f32_to_u32)
static_assert(2 * kSeqTiles * 16 * 255 * 255 < (1 << 23), "exact fp32 sums");

// This CTA's partial projection (reduced) from the workers' words; the caller
// synchronises before and after.
__device__ __forceinline__ void publish_partial(const SeqArgs &a, const SeqSmem &sm, int buf)
{
    u32 *dst = a.partial + ((size_t)buf * gridDim.x + blockIdx.x) * (kS * kS);
    if (threadIdx.x < kS * kS) {
        u64 tot = 0;
#pragma unroll
        for (int i = 0; i < kSeqWorkers; ++i) tot += sm.red[i][threadIdx.x];
        dst[threadIdx.x] = red64(tot, a.M);
    }
}

// S_step[o] = sum over CTAs of their partials (mod p), one warp per output:
// outputs blockIdx.x + gridDim.x (wi + k nw) for warp wi of nw.
__device__ void reduce_step(const SeqArgs &a, long long step, int wi, int nw)
{
    const int nb = gridDim.x;
    const int lane = threadIdx.x & 31;
    const u32 *src = a.partial + (size_t)(step % kSeqBufs) * nb * (kS * kS);
    for (int o = blockIdx.x + wi * nb; o < kS * kS; o += nb * nw) {
        u64 s = 0;
        for (int c = lane; c < nb; c += 32) s += __ldcg(src + (size_t)c * (kS * kS) + o);
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        const int ai = o / kS, bi = o % kS;
        if (lane == 0 && ai < a.s && bi < a.s) a.S[(step * a.s + ai) * a.s + bi] = red64(s, a.M);
    }
}

__global__ void __launch_bounds__(kSeqThreads, 1) k_sequence(const __grid_constant__ SeqArgs a)
{
    extern __shared__ __align__(16) unsigned char seq_smem[];
    SeqSmem &sm = *reinterpret_cast<SeqSmem *>(seq_smem);
    unsigned char *seq_dyn = seq_smem + sizeof(SeqSmem);
    const long long nb = gridDim.x;
    // 16-row aligned slices: every group of 16 rows belongs to one warp
    const int r0 = (int)(((a.n * blockIdx.x / nb) >> 4) << 4);
    const int r1 = blockIdx.x + 1 == nb ? (int)a.n : (int)(((a.n * (blockIdx.x + 1) / nb) >> 4) << 4);
    if (a.nsteps <= 0 && !a.Vnext) return;
    const int g0 = r0 >> 4, ng = (r1 - r0 + 15) >> 4, nr = r1 - r0;
    const uint4 *xf = a.XF + (size_t)g0 * 64;
    const u32 *col = a.col + r0, *val = a.val + r0;
    const unsigned char *gnp = a.gnp + g0;
    size_t ld = (size_t)a.ld;
    if (a.xf_smem) {
        // constant across steps: the CTA's X fragments
        uint4 *d = reinterpret_cast<uint4 *>(seq_dyn);
        for (int t = threadIdx.x; t < ng * 64; t += kSeqThreads) d[t] = __ldg(xf + t);
        xf = d;
    }
    if (a.mat_smem) {
        // constant across steps too: the CTA's rows of the matrix
        const int R = a.mrows;
        u32 *dc = reinterpret_cast<u32 *>(seq_dyn + a.mat_off), *dv = dc + (size_t)2 * a.npair * R;
        unsigned char *dg = reinterpret_cast<unsigned char *>(dv + (size_t)a.npair * R);
        for (int t = threadIdx.x; t < 2 * a.npair * nr; t += kSeqThreads) {
            const int e = t / nr, r = t - e * nr;
            dc[e * R + r] = __ldg(col + (size_t)e * ld + r);
        }
        for (int t = threadIdx.x; t < a.npair * nr; t += kSeqThreads) {
            const int e = t / nr, r = t - e * nr;
            dv[e * R + r] = __ldg(val + (size_t)e * ld + r);
        }
        for (int t = threadIdx.x; t < ng; t += kSeqThreads) dg[t] = __ldg(gnp + t);
        col = dc;
        val = dv;
        gnp = dg;
        ld = (size_t)R;
    }
    __syncthreads();
    const bool skip = a.test_skip && blockIdx.x == 0;
    const bool worker = threadIdx.x < 32 * kSeqWorkers;
    const u32 mu = (u32)(a.M.mu >> 32);   // floor(2^32 / m)
    // few CTAs have many outputs each: then every warp takes some
    const bool alone = kS * kS <= 3 * nb;
    const int wi = alone ? 0 : (int)(threadIdx.x >> 5), nw = alone ? 1 : kSeqWarps;
    unsigned epoch = 0;  // grid barriers passed
    // S_0 = X^T Y
    if (a.nsteps > 0) {
        if (worker) {
            const int last = seq_rows<false>(a, sm, xf, col, val, gnp, ld, a.V0, a.V0, r0, r1, true, mu);
            seq_project(a, sm, xf, last, ng, last < kSeqWorkers, mu);
        }
        __syncthreads();
        publish_partial(a, sm, 0);
        grid_arrive(a, skip);
        if (!grid_wait(a, skip, ++epoch)) return;
    }
    // Step i forms V_{i+1} and S_{i+1}'s partials.  These are written after
    // this CTA has arrived at the step's barrier, so they are seen after the
    // next one and summed in step i + 2; a buffer is written again only after
    // every CTA has arrived at the end of that step (kSeqBufs = 3).
    const long long steps = a.Vnext ? a.nsteps : a.nsteps - 1;   // products
    for (long long i = 0; i < steps; ++i) {
        const unsigned short *Vin = (i & 1) ? a.V1 : a.V0;
        unsigned short *Vout = (i & 1) ? a.V0 : a.V1;
        const bool proj = i + 1 < a.nsteps;
        if (i > 0 && (!worker || !alone)) reduce_step(a, i - 1, wi, nw);
        int last = 0;
        if (worker) last = seq_rows<true>(a, sm, xf, col, val, gnp, ld, Vin, Vout, r0, r1, proj, mu);
        grid_arrive(a, false);   // V_{i+1} is stored: the rest runs while the other CTAs arrive
        if (proj) {
            if (worker) seq_project(a, sm, xf, last, ng, last < kSeqWorkers, mu);
            __syncthreads();
            publish_partial(a, sm, (int)((i + 1) % kSeqBufs));
        }
        if (!grid_wait(a, false, ++epoch)) return;
    }
    // the last partials have to be seen, then the last two steps are summed
    if (a.nsteps > 1 && steps > 0) {
        grid_arrive(a, false);
        if (!grid_wait(a, false, ++epoch)) return;
    }
    for (long long j = steps > 1 ? steps - 1 : 0; j < a.nsteps; ++j)
        reduce_step(a, j, (int)(threadIdx.x >> 5), kSeqWarps);
    if (a.Vnext) {
        const unsigned short *Vf = (steps & 1) ? a.V1 : a.V0;
        for (long long t = (long long)r0 * a.s + threadIdx.x; t < (long long)r1 * a.s; t += kSeqThreads) {
            const long long row = t / a.s;
            const int c = (int)(t - row * a.s);
            a.Vnext[t] = __ldcg(Vf + row * kS + c);
        }
    }
}

// Y (n x s, u32) -> V0 (n x 16, u16, zero padded, reduced mod p).
__global__ void k_seq_prepare_v(long long n, int s, const u32 *__restrict__ Y,
                                unsigned short *V0, const Mod M)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * kS) return;
    const long long row = t / kS;
    const int c = (int)(t - row * kS);
    V0[t] = (unsigned short)(c < s ? red64(Y[row * s + c], M) : 0u);
}

// X (n x s, u32) -> its 8-bit limbs in m16n8k16 A-fragment order: for the
// 16-row group q, limb l and lane (g = lane/4, t = lane%4) the four f16x2
// words hold A[g][2t..2t+1], A[g+8][2t..2t+1], A[g][2t+8..9], A[g+8][2t+8..9]
// with A[a][k] = limb l of X[16q + k][a] (rows past n are zero).
__global__ void k_seq_prepare_x(long long n, int s, const u32 *__restrict__ X, uint4 *XF,
                                const Mod M)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nq = (n + 15) / 16;
    if (t >= nq * 2 * 32) return;
    const int lane = (int)(t & 31);
    const int l = (int)((t >> 5) & 1);
    const long long q = t >> 6;
    const int g = lane >> 2, tt = lane & 3;
    auto limb = [&](int k, int col) -> u32 {
        const long long row = q * 16 + k;
        if (row >= n || col >= s) return 0u;
        const u32 v = red64(X[row * s + col], M);
        return l ? (v >> 8) & 255u : v & 255u;
    };
    auto pair = [&](int k, int col) -> u32 {
        return bytes_to_half2(limb(k, col) | (limb(k + 1, col) << 16));
    };
    uint4 r;
    r.x = pair(2 * tt, g);
    r.y = pair(2 * tt, g + 8);
    r.z = pair(2 * tt + 8, g);
    r.w = pair(2 * tt + 8, g + 8);
    XF[t] = r;
}

// ---------------------------------------------------------------------------
// Per-launch path: projection S_step = X^T V (any p, s <= 32).
template <class Acc>
__global__ void __launch_bounds__(256) k_project(long long n, int s, const u32 *__restrict__ X,
                                                 const u32 *__restrict__ V, u64 *__restrict__ Sacc,
                                                 const Mod M)
{
    const int outs = s * s;
    for (int o = threadIdx.x; o < outs; o += blockDim.x) {
        const int ai = o / s, bi = o % s;
        Acc acc;
        acc.zero();
        for (long long k = blockIdx.x; k < n; k += gridDim.x)
            acc.mad(__ldg(X + k * s + ai), __ldg(V + k * s + bi));
        u64 part = acc.partial(M);
        atomicAdd(Sacc + o, (u64)red64(part, M));
    }
}

__global__ void k_project_finish(int outs, u64 *Sacc, u32 *S, const Mod M)
{
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= outs) return;
    S[o] = red64(Sacc[o], M);
    Sacc[o] = 0;
}

// dst row i (ldd words) = src row i (lds words, the first s of them) mod m,
// zero past s
__global__ void k_reduce_copy(long long n, int s, const u32 *__restrict__ src, int lds, u32 *__restrict__ dst, int ldd,
                              const Mod M)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * ldd) return;
    const long long i = t / ldd;
    const int c = (int)(t - i * ldd);
    dst[t] = c < s ? red64(src[i * lds + c], M) : 0u;
}

}  // namespace

// ---------------------------------------------------------------------------
struct SeqState {
    // entry pairs, row by row
    bool layout_tried = false, layout_ok = false;
    long long n = 0;
    int npair = 0;
    long long ld = 0;
    void *arena = nullptr;
    const u32 *col = nullptr, *val = nullptr;
    const unsigned char *gnp = nullptr;
    // work buffers
    void *work = nullptr;
    size_t work_bytes = 0;
    uint4 *XF = nullptr;
    unsigned short *V0 = nullptr, *V1 = nullptr;
    u32 *partial = nullptr;
    unsigned *bar = nullptr;
    int nblocks = 0;
    // per-launch path buffers, and the steps it was asked for
    long long steps = 0;
    void *gwork = nullptr;
    size_t gwork_bytes = 0;
    // graph cache: the kernel arguments and the two input blocks that the
    // captured preparation launches read
    cudaGraphExec_t exec = nullptr;
    SeqArgs key;
    const u32 *key_X = nullptr, *key_Y = nullptr;
};

void free_sequence_state(ffspmv_handle *h)
{
    SeqState *q = (SeqState *)h->seq_state;
    if (!q) return;
    if (q->exec) cudaGraphExecDestroy(q->exec);
    if (q->arena) cudaFree(q->arena);
    if (q->work) cudaFree(q->work);
    if (q->gwork) cudaFree(q->gwork);
    delete q;
    h->seq_state = nullptr;
}

namespace {

// The rows as pairs of entries: the densest diagonals first (their entries
// merged), then the rest in order.  Refused when a row needs more than kMaxEnt.
bool build_seq_layout(ffspmv_handle *h, SeqState &q)
{
    const long long n = h->A.nrows;
    const long long *ptr = h->h_ptr.data();
    const int *col = h->h_col.data();
    const u32 *val = h->h_val.data();
    std::vector<long long> cnt((size_t)(2 * n + 1), 0);
    for (long long i = 0; i < n; ++i)
        for (long long k = ptr[i]; k < ptr[i + 1]; ++k) cnt[(size_t)(col[k] - i + n)]++;
    std::vector<std::pair<long long, int>> cand;
    for (size_t t = 0; t < cnt.size(); ++t) {
        long long off = (long long)t - n;
        long long len = n - (off < 0 ? -off : off);
        if (cnt[t] && len * 4 >= n && cnt[t] * 2 >= len) cand.push_back({cnt[t], (int)off});
    }
    std::sort(cand.begin(), cand.end(), [](auto &x, auto &y) { return x.first > y.first; });
    std::vector<int> diag;
    for (size_t i = 0; i < cand.size() && i < 8; ++i) diag.push_back(cand[i].second);
    std::sort(diag.begin(), diag.end());
    const long long ld = (n + 31) / 32 * 32;
    std::vector<unsigned short> dval(diag.size() * ld, 0);
    std::vector<long long> rest(n, 0);
    long long width = 0;
    for (long long i = 0; i < n; ++i) {
        for (long long k = ptr[i]; k < ptr[i + 1]; ++k) {
            long long off = col[k] - i;
            auto it = std::find(diag.begin(), diag.end(), (int)off);
            if (it != diag.end()) {
                size_t idx = (size_t)(it - diag.begin()) * ld + i;
                dval[idx] = (unsigned short)(((u64)dval[idx] + val[k]) % h->m);
            } else {
                rest[i]++;
            }
        }
        width = std::max(width, rest[i]);
    }
    if (width + (long long)diag.size() > kMaxEnt) return false;  // short rows only
    if (n * kS >= (1LL << 31) || width * ld >= (1LL << 31)) return false;  // 32-bit indices
    const int nd = (int)diag.size(), npair = (int)((nd + width + 1) / 2);
    std::vector<u32> ecol((size_t)2 * npair * ld), eval((size_t)npair * ld, 0);
    std::vector<unsigned char> gnp((size_t)(n + 15) / 16, 0);
    for (size_t e = 0; e < (size_t)2 * npair; ++e)
        for (long long i = 0; i < ld; ++i) ecol[e * ld + i] = (u32)std::min<long long>(i, n - 1);
    for (long long i = 0; i < n; ++i) {
        int j = 0;   // entries without a value are left out
        auto put = [&](long long c, u32 v) {
            if (!v) return;
            ecol[(size_t)j * ld + i] = (u32)c;
            eval[(size_t)(j / 2) * ld + i] |= ((v & 255u) | (v >> 8) << 16) << (j & 1 ? 8 : 0);
            ++j;
        };
        for (int d = 0; d < nd; ++d) put(i + diag[d], dval[(size_t)d * ld + i]);
        for (long long k = ptr[i]; k < ptr[i + 1]; ++k)
            if (std::find(diag.begin(), diag.end(), (int)(col[k] - i)) == diag.end()) put(col[k], val[k]);
        unsigned char &g = gnp[(size_t)(i >> 4)];
        g = (unsigned char)std::max<int>(g, (j + 1) / 2);
    }
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t o_val = al(ecol.size() * 4 + 4), o_gnp = o_val + al(eval.size() * 4 + 4), total = o_gnp + al(gnp.size() + 4);
    if (cudaMalloc(&q.arena, total) != cudaSuccess) {
        q.arena = nullptr;
        return false;
    }
    char *b = (char *)q.arena;
    cudaMemcpy(b, ecol.data(), ecol.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(b + o_val, eval.data(), eval.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(b + o_gnp, gnp.data(), gnp.size(), cudaMemcpyHostToDevice);
    q.n = n;
    q.npair = npair;
    q.ld = ld;
    q.col = (const u32 *)b;
    q.val = (const u32 *)(b + o_val);
    q.gnp = (const unsigned char *)(b + o_gnp);
    return cudaGetLastError() == cudaSuccess;
}

ffspmv_status ensure_work(SeqState &q, long long n, int nblocks)
{
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t nq = (size_t)((n + 15) / 16);
    size_t xb = al(nq * 64 * sizeof(uint4));
    size_t vb = al((size_t)n * kS * 2 + 16);
    size_t pb = al((size_t)kSeqBufs * nblocks * kS * kS * 4);
    size_t need = xb + 2 * vb + pb + 256;
    if (need > q.work_bytes) {
        if (q.work) cudaFree(q.work);
        q.work = nullptr;
        q.work_bytes = 0;
        if (cudaMalloc(&q.work, need) != cudaSuccess) return FFSPMV_ERR_OOM;
        q.work_bytes = need;
    }
    char *b = (char *)q.work;
    q.XF = (uint4 *)b;
    q.V0 = (unsigned short *)(b + xb);
    q.V1 = (unsigned short *)(b + xb + vb);
    q.partial = (u32 *)(b + xb + 2 * vb);
    q.bar = (unsigned *)(b + xb + 2 * vb + pb);
    q.nblocks = nblocks;
    return FFSPMV_OK;
}

ffspmv_status sequence_per_launch(ffspmv_handle *h, SeqState &q, const u32 *X, const u32 *Y,
                                  int s, long long nsteps, u32 *S, u32 *Vnext, cudaStream_t st)
{
    const long long n = h->A.nrows;
    const Mod M = make_mod(h->m, 1, 0);
    // m > 2^16 and a format of the library's choice: one launch per step on the
    // block layout (4 001 rows, s = 8, p = 2^31 - 1: 5.2 us per step against
    // 17 with a projection, its finish and the plan's product).  The layout
    // has to be there or worth building: that takes 0.4 ms at 4 000 rows, 12 ms at
    // a million, what 20 to 60 steps gain (s = 1 to 16).  Steps of earlier calls
    // count (a sequence resumed piece by piece)
    const BlockPlan *B = nullptr;
    q.steps = std::min<long long>(q.steps + nsteps, 1LL << 40);
    if (h->m > 65536u && n > 0 && h->opt.sequence_mode == 0 && h->opt.priority_format == FFSPMV_FMT_AUTO &&
        nsteps > 0 && !(h->opt.test_hooks & 12) && (h->block[0] || q.steps >= kSeqBuildSteps))
        B = ensure_block(h, false, nullptr, 0, 0, st);
    int ldv = s;
    size_t vb = 0;
    for (;;) {
        ldv = B ? (s + 3) / 4 * 4 : s;
        vb = ((size_t)n * ldv * 4 + 255) / 256 * 256 + 256;
        const size_t need = 2 * vb + std::max((size_t)s * s * 8, B ? block_steps_bytes(n, s) : 0) + 256;
        if (need <= q.gwork_bytes) break;
        if (q.gwork) cudaFree(q.gwork);
        q.gwork = nullptr;
        q.gwork_bytes = 0;
        const bool deny = B && (h->opt.test_hooks & 32);   // testing
        if (!deny && cudaMalloc(&q.gwork, need) == cudaSuccess) {
            q.gwork_bytes = need;
            break;
        }
        cudaGetLastError();
        q.gwork = nullptr;
        if (!B) return FFSPMV_ERR_OOM;
        B = nullptr;   // the layout's steps take up to four times the rows of V at s < 4: without it, then
    }
    u32 *V[2] = {(u32 *)q.gwork, (u32 *)((char *)q.gwork + vb)};
    u64 *Sacc = (u64 *)((char *)q.gwork + 2 * vb);
    FF_CUDA(cudaMemsetAsync(Sacc, 0, (size_t)s * s * 8, st));
    if (n > 0) {
        k_reduce_copy<<<(unsigned)((n * ldv + 255) / 256), 256, 0, st>>>(n, s, Y, s, V[0], ldv, M);
        FF_CUDA(cudaGetLastError());
    }
    if (B) {
        // the product writes s words of every row of V_1: zero the rest once
        if (ldv != s) FF_CUDA(cudaMemsetAsync(V[1], 0, (size_t)n * ldv * 4, st));
        const ffspmv_status r = run_block_steps(*B, n, s, h->m, X, V[0], V[1], (u32 *)Sacc, nsteps, Vnext != nullptr,
                                                S, st);
        if (r != FFSPMV_OK) return r;
        if (Vnext) {
            k_reduce_copy<<<(unsigned)((n * s + 255) / 256), 256, 0, st>>>(n, s, V[nsteps & 1], ldv, Vnext, s, M);
            FF_CUDA(cudaGetLastError());
        }
        FF_CUDA(cudaStreamSynchronize(st));
        return FFSPMV_OK;
    }
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const unsigned pg = (unsigned)std::max<long long>(1, std::min<long long>(n, (long long)nsm));
    const int outs = s * s;
    const bool wide = (unsigned long long)(h->m - 1) * (h->m - 1) >
                      (~0ull) / (unsigned long long)std::max<long long>(n, 1);
    for (long long i = 0; i < nsteps; ++i) {
        const u32 *Vi = V[i & 1];
        if (n > 0) {
            if (wide)
                k_project<AccWide><<<pg, 256, 0, st>>>(n, s, X, Vi, Sacc, M);
            else
                k_project<AccSmall><<<pg, 256, 0, st>>>(n, s, X, Vi, Sacc, M);
            FF_CUDA(cudaGetLastError());
        }
        k_project_finish<<<(outs + 255) / 256, 256, 0, st>>>(outs, Sacc, S + i * outs, M);
        FF_CUDA(cudaGetLastError());
        if (i + 1 < nsteps || Vnext) {
            ffspmv_status r = run_plan(h->A, Vi, s, V[(i + 1) & 1], s, s, h->m, 1, 0, st);
            if (r != FFSPMV_OK) return r;
        }
    }
    if (Vnext && n > 0) {
        FF_CUDA(cudaMemcpyAsync(Vnext, V[nsteps & 1], (size_t)n * s * 4,
                                cudaMemcpyDeviceToDevice, st));
    }
    FF_CUDA(cudaStreamSynchronize(st));
    return FFSPMV_OK;
}

bool same_key(const SeqArgs &a, const SeqArgs &b)
{
    return memcmp(&a, &b, sizeof(SeqArgs)) == 0;
}

}  // namespace

}  // namespace ff

using namespace ff;

extern "C" ffspmv_status spmv_block_sequence(ffspmv_t h, const uint32_t *d_X, const uint32_t *d_Y,
                                             int32_t s, int64_t start_step, int64_t nsteps,
                                             uint32_t *d_S, uint32_t *d_V_state,
                                             ffspmv_stream_t stream)
{
    if (!h || s < 1 || s > 32 || nsteps < 0 || start_step < 0) return FFSPMV_ERR_ARG;
    if (h->A.nrows != h->A.ncols) return FFSPMV_ERR_ARG;
    const long long n = h->A.nrows;
    // a resumed sequence starts from the state an earlier call left in d_V_state
    if (start_step > 0 && !d_V_state) return FFSPMV_ERR_ARG;
    if (start_step > 0) d_Y = d_V_state;
    uint32_t *d_V_next = d_V_state;
    if (n > 0 && (!d_X || !d_Y)) return FFSPMV_ERR_ARG;
    if (nsteps > 0 && !d_S) return FFSPMV_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (!h->seq_state) h->seq_state = new (std::nothrow) SeqState();
    SeqState *q = (SeqState *)h->seq_state;
    if (!q) return FFSPMV_ERR_OOM;

    bool persistent = h->opt.sequence_mode == 0 && h->m <= 65536u && s <= kS && n > 0 && nsteps > 0;
    if (persistent && !q->layout_tried) {
        q->layout_tried = true;
        q->layout_ok = build_seq_layout(h, *q);
    }
    persistent = persistent && q->layout_ok;
    int nblocks = 0;
    if (persistent) {
        int dev = 0, nsm = 0, per_sm = 0, coop = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        cudaFuncSetAttribute(k_sequence, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(SeqSmem) + kXfSmemMax));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sequence, kSeqThreads, sizeof(SeqSmem) + kXfSmemMax);
        nblocks = nsm * std::min(per_sm, 1);
        if (!coop || per_sm < 1) persistent = false;
        // keep at least one pass of rows per CTA
        long long maxb = std::max<long long>(1, n / 16);
        if (nblocks > maxb) nblocks = (int)maxb;
    }
    if (!persistent) return sequence_per_launch(h, *q, d_X, d_Y, s, nsteps, d_S, d_V_next, st);

    ffspmv_status rs = ensure_work(*q, n, nblocks);
    if (rs != FFSPMV_OK) return rs;
    SeqArgs a;
    memset(&a, 0, sizeof(a));
    a.n = n;
    a.npair = q->npair;
    a.s = s;
    a.ld = q->ld;
    a.nsteps = nsteps;
    a.col = q->col;
    a.val = q->val;
    a.gnp = q->gnp;
    a.XF = q->XF;
    a.V0 = q->V0;
    a.V1 = q->V1;
    a.partial = q->partial;
    a.S = d_S;
    a.Vnext = d_V_next;
    a.bar = q->bar;
    a.status = h->d_status;
    a.spin_limit = h->opt.barrier_spin_limit ? h->opt.barrier_spin_limit : kDefaultSpins;
    a.test_skip = (h->opt.test_hooks & 1) ? 1 : 0;
    // X fragments of the largest CTA slice: 1 KB per 16-row group (+ 2 groups of rounding)
    const size_t xf_bytes = (size_t)((n + nblocks - 1) / nblocks / 16 + 2) * 64 * sizeof(uint4);
    a.xf_smem = xf_bytes <= kXfSmemMax ? 1 : 0;
    // the CTA's matrix rows as well, when they fit beside the X fragments
    a.mrows = (int)(((n + nblocks - 1) / nblocks / 16 + 2) * 16);
    const size_t mat_bytes = (size_t)3 * q->npair * a.mrows * 4 + (size_t)a.mrows / 16 + 16;
    a.mat_off = a.xf_smem ? (int)xf_bytes : 0;
    a.mat_smem = (size_t)a.mat_off + mat_bytes <= kXfSmemMax ? 1 : 0;
    const size_t dyn_smem = sizeof(SeqSmem) + (size_t)a.mat_off + (a.mat_smem ? mat_bytes : 0);
    a.M = make_mod(h->m, 1, 0);

    // the graph: prepare X/Y, clear barrier + status, run the persistent kernel
    if (!q->exec || !same_key(a, q->key) || q->key_X != d_X || q->key_Y != d_Y) {
        if (q->exec) cudaGraphExecDestroy(q->exec);
        q->exec = nullptr;
        cudaStream_t cs;
        FF_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaGraph_t g = nullptr;
        bool ok = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
        if (ok) {
            const long long nxf = (n + 15) / 16 * 64;
            k_seq_prepare_x<<<(unsigned)((nxf + 255) / 256), 256, 0, cs>>>(n, s, d_X, q->XF, a.M);
            k_seq_prepare_v<<<(unsigned)((n * kS + 255) / 256), 256, 0, cs>>>(n, s, d_Y, q->V0, a.M);
            cudaMemsetAsync(q->bar, 0, 2 * sizeof(unsigned), cs);
            cudaMemsetAsync(h->d_status, 0, sizeof(int), cs);
            cudaLaunchConfig_t cfg;
            memset(&cfg, 0, sizeof(cfg));
            cfg.gridDim = dim3((unsigned)nblocks);
            cfg.blockDim = dim3(kSeqThreads);
            cfg.dynamicSmemBytes = dyn_smem;
            cfg.stream = cs;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeCooperative;
            at[0].val.cooperative = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            cudaError_t le = cudaLaunchKernelEx(&cfg, k_sequence, a);
            cudaError_t ce = cudaStreamEndCapture(cs, &g);
            ok = le == cudaSuccess && ce == cudaSuccess && g != nullptr;
            if (ok) ok = cudaGraphInstantiate(&q->exec, g, 0) == cudaSuccess;
            if (g) cudaGraphDestroy(g);
        }
        cudaGetLastError();
        cudaStreamDestroy(cs);
        if (!ok) {
            q->exec = nullptr;
            return sequence_per_launch(h, *q, d_X, d_Y, s, nsteps, d_S, d_V_next, st);
        }
        q->key = a;
        q->key_X = d_X;
        q->key_Y = d_Y;
    }
    FF_CUDA(cudaGraphLaunch(q->exec, st));
    int status = 0;
    FF_CUDA(cudaMemcpyAsync(&status, h->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
    FF_CUDA(cudaStreamSynchronize(st));
    if (status != 0) {
        cudaMemset(h->d_status, 0, sizeof(int));
        return FFSPMV_ERR_TIMEOUT;
    }
    return FFSPMV_OK;
}

// The projection of one step on its own, for a sequence whose rows are split
// over several processes: each adds its rows' X^T V into a u64 accumulator,
// the accumulators are summed across processes, and the finish reduces them.
extern "C" ffspmv_status spmv_block_project(uint32_t p, int64_t n, int32_t s, const uint32_t *d_X,
                                            const uint32_t *d_V, uint64_t *d_Sacc, ffspmv_stream_t stream)
{
    if (p < 2 || n < 0 || s < 1 || s > 32 || !d_Sacc || (n > 0 && (!d_X || !d_V))) return FFSPMV_ERR_ARG;
    if (n == 0) return FFSPMV_OK;
    const Mod M = make_mod(p, 1, 0);
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const unsigned pg = (unsigned)std::max<long long>(1, std::min<long long>(n, (long long)std::max(nsm, 1)));
    const bool wide = (unsigned long long)(p - 1) * (p - 1) > (~0ull) / (unsigned long long)n;
    if (wide)
        k_project<AccWide><<<pg, 256, 0, st>>>(n, s, d_X, d_V, (u64 *)d_Sacc, M);
    else
        k_project<AccSmall><<<pg, 256, 0, st>>>(n, s, d_X, d_V, (u64 *)d_Sacc, M);
    FF_CUDA(cudaGetLastError());
    return FFSPMV_OK;
}

extern "C" ffspmv_status spmv_block_project_finish(uint32_t p, int32_t s, uint64_t *d_Sacc, uint32_t *d_S,
                                                   ffspmv_stream_t stream)
{
    if (p < 2 || s < 1 || s > 32 || !d_Sacc || !d_S) return FFSPMV_ERR_ARG;
    const Mod M = make_mod(p, 1, 0);
    const int outs = s * s;
    k_project_finish<<<(outs + 255) / 256, 256, 0, (cudaStream_t)stream>>>(outs, (u64 *)d_Sacc, d_S, M);
    FF_CUDA(cudaGetLastError());
    return FFSPMV_OK;
}
