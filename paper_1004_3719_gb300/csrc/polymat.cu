// Products of s x s polynomial matrices over Z/pZ, C(x) = A(x) B(x): the
// multiplication that the sigma-basis / PM-Basis step of block Wiedemann is
// built from, by the fast algorithm of Sec. 3 (parallel polynomial matrix
// multiplication): evaluate both operands at the powers of a root of unity,
// multiply the matrices point by point, interpolate back.  Coefficient-major
// arrays: A[k][i][j] is the coefficient of x^k in entry (i, j).
//
// F_p itself has roots of unity of order at most 16 when p = 65521, so the
// transforms run over primes with large power-of-two roots instead: the
// exact integer coefficients of C are below s * (min(da, db) + 1) * (p-1)^2,
// so C is computed modulo as many primes as that bound needs (one, two or
// three: two for p = 65521 at every length, three for p near 2^31), by
// number-theoretic transforms of length L (a power of two >= da+db+1), a
// pointwise matrix product at each of the L points, and the inverse
// transforms, then brought back to Z/pZ by Garner's mixed-radix
// reconstruction.
//
// Layout.  Every array stays point-major, [prime][point][entry]: the entries
// of one matrix are contiguous, like the coefficients that come in and go
// out.  A transform works on all entries at once, one (entry, column) item
// per lane, so that every global access of a warp is 32 consecutive words
// whatever the matrix size; nothing is transposed.  L = L1 L2: a first
// kernel transforms along k1 (k = k1 L2 + k2, stride L2) and multiplies by
// the cross twiddles w^(j1 k2), a second along k2; the inverse runs the same
// two axes backwards, so the frequencies are never reordered.  L <= 256
// takes one kernel each way.  One tile is up to 256 points x 32 items: two
// register transforms of up to 16 points per thread with one exchange
// through shared memory between them.
//
// What bounds it: at s = 16, degree 6250 (L = 16384, two primes) the planes
// of A, B and C are 33.5 MB each, and each is written and read twice; the
// butterflies (about 7 instructions each on values kept in [0, 2P)) are the
// rest.  Measured with the former one-polynomial-per-CTA radix-2 kernels over
// three primes: 1170 us per product; with these: 148 us.
#include <algorithm>
#include <cstring>

#include "ff_internal.cuh"
#include "ff_polymat.h"
#include "ffspmv_polymat.h"

namespace ff {
namespace {

constexpr int kPmPrimes = 3;
constexpr u32 kPmP0 = 998244353u, kPmP1 = 469762049u, kPmP2 = 167772161u;  // c 2^k + 1, k = 23, 26, 25
constexpr u32 kPmP[kPmPrimes] = {kPmP0, kPmP1, kPmP2};
constexpr u32 kPmGen = 3;                                            // a primitive root of each
constexpr int kPmMaxLog = 15;
constexpr int kPmMinLog = 4;
constexpr int kPmLanes = 32;                                         // items per tile

// ---------------------------------------------------------------------------
// Roots of unity, computed by the compiler.
struct alignas(8) PmW {
    u32 w, q;  // a constant and floor(w 2^32 / P), its Shoup quotient
};

constexpr u32 pm_pow(u64 a, u64 e, u64 m)
{
    u64 r = 1 % m;
    a %= m;
    while (e) {
        if (e & 1) r = r * a % m;   // m < 2^30
        a = a * a % m;
        e >>= 1;
    }
    return (u32)r;
}

constexpr u32 pm_inv32(u32 m)  // m^-1 mod 2^32, m odd (Newton)
{
    u32 y = m;
    for (int i = 0; i < 4; ++i) y *= 2u - m * y;
    return y;
}

constexpr u32 pm_root(int q, int lg) { return pm_pow(kPmGen, (kPmP[q] - 1) >> lg, kPmP[q]); }

constexpr PmW pm_w(u64 w, u64 P) { return PmW{(u32)w, (u32)((w << 32) / P)}; }

struct PmConstTab {
    PmW w16[2][kPmPrimes][8];     // powers of the 16th root and of its inverse
    PmW w256[kPmPrimes][256];     // powers of the 256th root
};

constexpr PmConstTab pm_make_const()
{
    PmConstTab t{};
    for (int q = 0; q < kPmPrimes; ++q) {
        const u64 P = kPmP[q];
        for (int dir = 0; dir < 2; ++dir) {
            const u64 r = dir ? pm_pow(pm_root(q, 4), P - 2, P) : pm_root(q, 4);
            u64 w = 1;
            for (int i = 0; i < 8; ++i) {
                t.w16[dir][q][i] = pm_w(w, P);
                w = w * r % P;
            }
        }
        u64 w = 1;
        const u64 r = pm_root(q, 8);
        for (int i = 0; i < 256; ++i) {
            t.w256[q][i] = pm_w(w, P);
            w = w * r % P;
        }
    }
    return t;
}

// Powers of the 2^15-th root w in Montgomery form: w^(256 h) at hi[h], w^l at
// lo[l]; w^i is the Montgomery product of two entries.
struct PmCrossTab {
    u32 hi[kPmPrimes][128], lo[kPmPrimes][256];
};

constexpr PmCrossTab pm_make_cross()
{
    PmCrossTab t{};
    for (int q = 0; q < kPmPrimes; ++q) {
        const u64 P = kPmP[q], R = ((u64)1 << 32) % P;
        u64 w = R, r = pm_root(q, 7);
        for (int i = 0; i < 128; ++i) {
            t.hi[q][i] = (u32)w;
            w = w * r % P;
        }
        w = R;
        r = pm_root(q, 15);
        for (int i = 0; i < 256; ++i) {
            t.lo[q][i] = (u32)w;
            w = w * r % P;
        }
    }
    return t;
}

__constant__ const PmConstTab c_pm = pm_make_const();
__device__ const PmCrossTab d_pm_cross = pm_make_cross();

// ---------------------------------------------------------------------------
// Arithmetic mod P < 2^30 on lazy values in [0, 2P).
__device__ __forceinline__ u32 pm_csub(u32 x, u32 m) { return min(x, x - m); }  // x < 2m: x mod m up to m

// a w mod P in [0, 2P) for any 32-bit a and a fixed w < P (Shoup): the
// quotient estimate umulhi(a, q) is the true quotient or one less.
__device__ __forceinline__ u32 pm_shoup(u32 a, u32 w, u32 q, u32 P) { return a * w - __umulhi(a, q) * P; }

// hi 2^32 + lo, times 2^-32, mod P (Montgomery, 1985): in [0, P + hi] without
// overflow when hi + P < 2^32.
__device__ __forceinline__ u32 pm_redc(u32 lo, u32 hi, u32 P, u32 pinv) { return hi + P - __umulhi(lo * pinv, P); }

// a b 2^-32 mod P in [0, 2P), for a < 2^32 and b < P
__device__ __forceinline__ u32 pm_mont(u32 a, u32 b, u32 P, u32 pinv)
{
    const u64 t = (u64)a * b;
    return pm_redc((u32)t, (u32)(t >> 32), P, pinv);
}

struct PmPrime {
    u32 P, pinv, mu;  // mu = floor(2^32 / P)
};

__device__ __forceinline__ PmPrime pm_prime(int q)
{
    PmPrime r;
    r.P = q == 0 ? kPmP0 : q == 1 ? kPmP1 : kPmP2;
    constexpr u32 i0 = pm_inv32(kPmP0), i1 = pm_inv32(kPmP1), i2 = pm_inv32(kPmP2);
    constexpr u32 m0 = (u32)(((u64)1 << 32) / kPmP0), m1 = (u32)(((u64)1 << 32) / kPmP1),
                  m2 = (u32)(((u64)1 << 32) / kPmP2);
    r.pinv = q == 0 ? i0 : q == 1 ? i1 : i2;
    r.mu = q == 0 ? m0 : q == 1 ? m1 : m2;
    return r;
}

// v < 2^bits with its bits reversed, bits <= 4
__host__ __device__ constexpr int pm_bitrev(int v, int bits)
{
    return ((v & 1) << 3 | (v & 2) << 1 | (v & 4) >> 1 | (v & 8) >> 3) >> (4 - bits);
}

// Stages ST, ST - 1, ..., 0 of a decimation in frequency over 2^LOG points in
// registers: X_j ends at register bitrev(j).  Values in and out in [0, 2P).
template <int LOG, int ST, bool INV>
__device__ __forceinline__ void pm_stages(u32 (&x)[1 << LOG], int q, u32 P)
{
    constexpr int len = 1 << ST;
    const u32 P2 = 2u * P;
#pragma unroll
    for (int h = 0; h < (1 << LOG) / 2; ++h) {
        const int i = h & (len - 1), k = ((h >> ST) << (ST + 1)) + i;
        const u32 u = x[k], v = x[k + len], d = u - v + P2;
        x[k] = pm_csub(u + v, P2);
        if (i == 0) {
            x[k + len] = pm_csub(d, P2);
        } else {
            const PmW w = c_pm.w16[INV ? 1 : 0][q][i * (8 >> ST)];
            x[k + len] = pm_shoup(d, w.w, w.q, P);
        }
    }
    if constexpr (ST > 0) pm_stages<LOG, ST - 1, INV>(x, q, P);
}

template <int LOG, bool INV>
__device__ __forceinline__ void pm_dft(u32 (&x)[1 << LOG], int q, u32 P)
{
    pm_stages<LOG, LOG - 1, INV>(x, q, P);
}

// The tile transform of 2^(LA+LB) points for one lane's item: x holds points
// n = na 2^LB + g (g the thread's group) on entry; on return y(r, jb) is
// frequency j = ja + 2^LA jb of ja = g + r 2^LB, at register
// r 2^LB + bitrev(jb).  `sm` is the tile's exchange buffer.
template <int LA, int LB, bool INV>
__device__ __forceinline__ void pm_tile(u32 (&x)[1 << LA], u32 *sm, int g, int lane, int q, u32 P)
{
    constexpr int NA = 1 << LA, NB = 1 << LB;
    static_assert(LA >= LB, "a group's step B takes NA / NB frequencies ja");
    pm_dft<LA, INV>(x, q, P);
#pragma unroll
    for (int ja = 0; ja < NA; ++ja) {
        u32 v = x[pm_bitrev(ja, LA)];
        if (ja) {
            const int e = (ja * g) << (8 - LA - LB);  // exponent of the 256th root
            const PmW w = c_pm.w256[q][INV ? (256 - e) & 255 : e];
            v = pm_shoup(v, w.w, w.q, P);
        }
        sm[(ja * NB + g) * kPmLanes + lane] = v;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < NA / NB; ++r) {
        u32 y[NB];
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) y[nb] = sm[((g + r * NB) * NB + nb) * kPmLanes + lane];
        pm_dft<LB, INV>(y, q, P);
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) x[r * NB + nb] = y[nb];
    }
}

// One operand of a transform launch: `ne` entries per point.
struct PmOp {
    const u32 *src;      // coefficients (first forward pass), else unused
    long long nsrc;      // words of src
    u32 *plane;          // [prime][L][ne]
    int ne;
    unsigned tiles;      // CTAs of this operand
};

enum PmMode { PM_F1, PM_F2, PM_F, PM_I1 };

// One pass over one axis of L = L1 L2 for one or two operands (blockIdx.x)
// and one prime (blockIdx.y).  PM_F1: along k1, coefficients in, times the
// cross twiddles; PM_F2: along k2, values out below P; PM_F: the only pass
// (L2 = 1), coefficients in, values out below P; PM_I1: inverse along j2,
// times the inverse cross twiddles.
template <int LA, int LB, int MODE>
__global__ void __launch_bounds__(kPmLanes << LB) k_pm_pass(const PmOp A, const PmOp B, int lg, int lg2)
{
    constexpr int NA = 1 << LA, NB = 1 << LB, LN = LA + LB;
    constexpr bool INV = MODE == PM_I1, FIRST = MODE == PM_F1 || MODE == PM_F;
    __shared__ u32 sm[(1 << LN) * kPmLanes];
    const bool isB = blockIdx.x >= A.tiles;
    const PmOp &O = isB ? B : A;
    const unsigned tile = isB ? blockIdx.x - A.tiles : blockIdx.x;
    const int q = blockIdx.y, lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const PmPrime pr = pm_prime(q);
    const u32 P = pr.P;
    const int ne = O.ne;
    // items: (k2, entry) along k1, (j1, entry) along k2
    const u32 other = 1u << (lg - LN);   // points of the other axis
    const u32 w = tile * kPmLanes + lane;
    const bool ok = w < other * (u32)ne;
    const u32 kk = w / (u32)ne;
    const u32 stride = FIRST ? ((u32)ne << lg2) : (u32)ne;
    const u32 base = FIRST ? w : kk * ((u32)ne << lg2) + (w - kk * (u32)ne);
    u32 *pl = O.plane + (size_t)q * ((size_t)ne << lg);
    u32 x[NA];
#pragma unroll
    for (int na = 0; na < NA; ++na) {
        const u32 n = (u32)(na * NB + g), idx = base + n * stride;
        x[na] = 0u;
        if (FIRST) {
            if (ok && (long long)idx < O.nsrc) {
                const u32 v = __ldg(O.src + idx);
                x[na] = v - __umulhi(v, pr.mu) * P;  // below 2P (Barrett, 1986)
            }
        } else if (ok) {
            x[na] = pl[idx];
        }
    }
    pm_tile<LA, LB, INV>(x, sm, g, lane, q, P);
    if (!ok) return;
    // cross twiddle of frequency j: the 2^15-th root to the power +-j kk 2^(15-lg),
    // Montgomery form; from one jb to the next it takes a fixed factor
    auto cross = [&](u32 e) {
        e = (INV ? (1u << kPmMaxLog) - e : e) & ((1u << kPmMaxLog) - 1u);
        return pm_csub(pm_mont(__ldg(&d_pm_cross.hi[q][e >> 8]), __ldg(&d_pm_cross.lo[q][e & 255u]), P, pr.pinv), P);
    };
    const u32 ke = kk << (kPmMaxLog - lg);
    const u32 step = (MODE == PM_F1 || MODE == PM_I1) ? cross(NA * ke) : 0u;
#pragma unroll
    for (int r = 0; r < NA / NB; ++r) {
        const u32 j0 = (u32)(g + r * NB);
        u32 t = (MODE == PM_F1 || MODE == PM_I1) ? cross(j0 * ke) : 0u;
#pragma unroll
        for (int jb = 0; jb < NB; ++jb) {
            u32 v = x[r * NB + pm_bitrev(jb, LB)];
            if (MODE == PM_F1 || MODE == PM_I1) {
                v = pm_mont(v, t, P, pr.pinv);
                if (jb + 1 < NB) t = pm_csub(pm_mont(t, step, P, pr.pinv), P);
            } else {
                v = pm_csub(v, P);
            }
            pl[base + (j0 + NA * jb) * stride] = v;
        }
    }
}

struct PmOut {
    Mod mp;                    // the output modulus p
    u32 linv[kPmPrimes], linv_q[kPmPrimes];  // 2^32 / L mod P and its Shoup quotient
    u32 inv01, inv01q, inv02, inv02q, inv12, inv12q;  // P0^-1 mod P1, mod P2, P1^-1 mod P2, with quotients
    u32 p0_mod_p, p0p1_mod_p;
};

// x mod P for x < 2^30 and P < 2^30 with mu = floor(2^32 / P)
__device__ __forceinline__ u32 pm_mod(u32 x, u32 P, u32 mu) { return pm_csub(x - __umulhi(x, mu) * P, P); }

// The integer with residues r[0..NPR-1] (each below its prime), mod p (Garner)
template <int NPR>
__device__ __forceinline__ u32 pm_crt(const u32 (&r)[NPR], const PmOut &c)
{
    if constexpr (NPR == 1) return red64(r[0], c.mp);
    if constexpr (NPR >= 2) {
        constexpr u32 P0 = kPmP0, P1 = kPmP1, P2 = kPmP2;
        constexpr u32 mu1 = (u32)(((u64)1 << 32) / P1), mu2 = (u32)(((u64)1 << 32) / P2);
        const u32 d1 = r[1] + P1 - pm_mod(r[0], P1, mu1);
        const u32 x2 = pm_csub(pm_shoup(d1, c.inv01, c.inv01q, P1), P1);
        if constexpr (NPR == 2) return red64((u64)r[0] + (u64)P0 * x2, c.mp);   // below P0 P1 < 2^59
        if constexpr (NPR == 3) {
            const u32 d2 = r[2] + P2 - pm_mod(r[0], P2, mu2);
            const u32 t2 = pm_csub(pm_shoup(d2, c.inv02, c.inv02q, P2), P2);
            const u32 d3 = t2 + P2 - pm_mod(x2, P2, mu2);
            const u32 x3 = pm_csub(pm_shoup(d3, c.inv12, c.inv12q, P2), P2);
            // r0 + P0 x2 + P0 P1 x3, term by term
            const u64 v = (u64)red64(r[0], c.mp) + red64((u64)c.p0_mod_p * x2, c.mp) + red64((u64)c.p0p1_mod_p * x3, c.mp);
            return red64(v, c.mp);
        }
    }
}

// The last inverse pass, along j1, for every prime in turn, then the
// reconstruction: coefficients klo..khi of C are written from C on.
template <int LA, int LB, int NPR>
__global__ void __launch_bounds__(kPmLanes << LB) k_pm_out(const u32 *__restrict__ Ch, u32 *__restrict__ C, int ne, int lg,
                                                          int lg2, long long klo, long long khi, const __grid_constant__ PmOut c)
{
    constexpr int NA = 1 << LA, NB = 1 << LB, LN = LA + LB;
    __shared__ u32 sm[(1 << LN) * kPmLanes];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const u32 w = blockIdx.x * kPmLanes + lane;
    const bool ok = w < ((u32)ne << (lg - LN));
    const u32 stride = (u32)ne << lg2;
    u32 res[NPR][NA];
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
        const u32 *pl = Ch + (size_t)q * ((size_t)ne << lg);
#pragma unroll
        for (int na = 0; na < NA; ++na) res[q][na] = ok ? pl[w + (u32)(na * NB + g) * stride] : 0u;
        if (q) __syncthreads();  // the previous prime's exchange has been read
        pm_tile<LA, LB, true>(res[q], sm, g, lane, q, pm_prime(q).P);
    }
    if (!ok) return;
    const long long lo = klo * ne, hi = (khi + 1) * ne;
#pragma unroll
    for (int r = 0; r < NA / NB; ++r)
#pragma unroll
        for (int jb = 0; jb < NB; ++jb) {
            const long long idx = w + (long long)(g + r * NB + NA * jb) * stride;
            if (idx < lo || idx >= hi) continue;
            u32 v[NPR];
#pragma unroll
            for (int q = 0; q < NPR; ++q)
                v[q] = pm_csub(pm_shoup(res[q][r * NB + pm_bitrev(jb, LB)], c.linv[q], c.linv_q[q], pm_prime(q).P), pm_prime(q).P);
            C[idx - lo] = pm_crt<NPR>(v, c);
        }
}

// ---------------------------------------------------------------------------
// Ch[q][t] = Ah[q][t] Bh[q][t] 2^-32 mod P_q, an (sr x si) by (si x sc) product
// at every point.  A CTA takes TP consecutive points of one prime, both
// matrices of each in shared memory (rows padded to four words); a thread
// forms 4 x 4 outputs of one point (rows ti + nti r, columns 4 tj ..), reading
// four words of four rows of A and of B at a time: 64 multiply-adds per eight
// 16-byte loads.  Terms are below P^2 < 2^59.8, so 16 of them fit in 64 bits;
// longer rows fold multiples of 2 P 2^32 away every eight terms.
constexpr int kPwThreads = 256;

struct PmPw {
    int sr, si, sc;
    int si4, sc4;        // si, sc rounded up to 4
    int nti, ntj;        // threads per point: rows (sr / 4), columns (sc / 4), rounded up
    int tp;              // points per CTA
    int ast, bst;        // words of shared memory per point of A and of B
    int L;
    u32 m_a, m_si, m_b, m_sc;  // ceil(2^32 / d) for d = sr si, si, si sc, sc: exact quotients below 2^16
};

__device__ __forceinline__ u32 pm_div(u32 x, u32 magic) { return __umulhi(x, magic); }

__global__ void __launch_bounds__(kPwThreads) k_pm_pointwise(const u32 *__restrict__ Ah, const u32 *__restrict__ Bh,
                                                            u32 *__restrict__ Ch, const __grid_constant__ PmPw a)
{
    extern __shared__ __align__(16) u32 pw[];
    u32 *As = pw, *Bs = pw + (size_t)a.tp * a.ast;
    const int q = blockIdx.y, t0 = blockIdx.x * a.tp, np = min(a.tp, a.L - t0);
    const PmPrime pr = pm_prime(q);
    const u32 ea = (u32)(a.sr * a.si), eb = (u32)(a.si * a.sc), ec = (u32)(a.sr * a.sc);
    const u32 *ag = Ah + ((size_t)q * a.L + t0) * ea, *bg = Bh + ((size_t)q * a.L + t0) * eb;
    // rows and columns past the matrices are never used but read: zero them
    if (a.si != a.si4 || a.sc != a.sc4 || a.sr != 4 * a.nti) {
        for (int i = threadIdx.x; i < a.tp * (a.ast + a.bst); i += kPwThreads) pw[i] = 0u;
        __syncthreads();
        for (u32 i = threadIdx.x; i < (u32)np * ea; i += kPwThreads) {
            const u32 t = ea == 1u ? i : pm_div(i, a.m_a), e = i - t * ea;
            const u32 r = a.si == 1 ? e : pm_div(e, a.m_si), k = e - r * (u32)a.si;
            As[t * a.ast + r * a.si4 + k] = ag[i];
        }
        for (u32 i = threadIdx.x; i < (u32)np * eb; i += kPwThreads) {
            const u32 t = eb == 1u ? i : pm_div(i, a.m_b), e = i - t * eb;
            const u32 r = a.sc == 1 ? e : pm_div(e, a.m_sc), k = e - r * (u32)a.sc;
            Bs[t * a.bst + r * a.sc4 + k] = bg[i];
        }
    } else {
        // multiples of four: whole 16-byte blocks (the planes are 16-byte aligned)
        for (u32 i = threadIdx.x; i < (u32)np * ea / 4; i += kPwThreads) {
            const u32 t = pm_div(4 * i, a.m_a);
            *reinterpret_cast<uint4 *>(As + t * a.ast + (4 * i - t * ea)) = reinterpret_cast<const uint4 *>(ag)[i];
        }
        for (u32 i = threadIdx.x; i < (u32)np * eb / 4; i += kPwThreads) {
            const u32 t = pm_div(4 * i, a.m_b);
            *reinterpret_cast<uint4 *>(Bs + t * a.bst + (4 * i - t * eb)) = reinterpret_cast<const uint4 *>(bg)[i];
        }
    }
    __syncthreads();
    const int per = a.nti * a.ntj, t = threadIdx.x / per, u = threadIdx.x - t * per;
    if (t >= np) return;
    const int ti = u / a.ntj, tj = u - ti * a.ntj;
    const u32 *ap = As + t * a.ast + ti * a.si4, *bp = Bs + t * a.bst + 4 * tj;
    u64 acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0;
    const u32 P2 = 2u * pr.P;
    for (int k = 0; k < a.si4; k += 4) {
        uint4 av[4], bv[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) av[r] = *reinterpret_cast<const uint4 *>(ap + r * a.nti * a.si4 + k);
#pragma unroll
        for (int r = 0; r < 4; ++r) bv[r] = *reinterpret_cast<const uint4 *>(bp + (k + r) * a.sc4);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const u32 ar[4] = {av[r].x, av[r].y, av[r].z, av[r].w};
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                acc[r][0] += (u64)ar[h] * bv[h].x;
                acc[r][1] += (u64)ar[h] * bv[h].y;
                acc[r][2] += (u64)ar[h] * bv[h].z;
                acc[r][3] += (u64)ar[h] * bv[h].w;
            }
        }
        if (a.si > 16 && (k & 4)) {
            // eight more terms add below 8 P^2 < 2^62.8 to at most 2 P 2^32 < 2^62.9
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const u32 h = (u32)(acc[r][c] >> 32);
                    acc[r][c] = (u64)min(h, h - P2) << 32 | (u32)acc[r][c];
                }
        }
    }
    u32 *cg = Ch + ((size_t)q * a.L + t0 + t) * ec;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = ti + r * a.nti;
        if (i >= a.sr) break;
        u32 o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            // the high word is below 3.8 P (16 terms) or 4P: one or two steps of 2P
            u32 h = (u32)(acc[r][c] >> 32);
            h = min(h, h - P2);
            const u32 v = pm_redc((u32)acc[r][c], h, pr.P, pr.pinv);   // below 3P
            o[c] = pm_csub(v, P2);
        }
        if (a.sc == a.sc4) {
            *reinterpret_cast<uint4 *>(cg + (size_t)i * a.sc + 4 * tj) = make_uint4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (4 * tj + c < a.sc) cg[(size_t)i * a.sc + 4 * tj + c] = o[c];
        }
    }
}

int pm_log2(long long points)
{
    int lg = kPmMinLog;
    while ((1LL << lg) < points) ++lg;
    return lg;
}

// Launches of one axis of 2^ln points (4 <= ln <= 8).
template <int MODE>
ffspmv_status pm_pass(int ln, const PmOp &A, const PmOp &B, int lg, int lg2, int npr, cudaStream_t st)
{
    const dim3 grid(A.tiles + B.tiles, (unsigned)npr);
    switch (ln) {
    case 4: k_pm_pass<2, 2, MODE><<<grid, kPmLanes << 2, 0, st>>>(A, B, lg, lg2); break;
    case 5: k_pm_pass<3, 2, MODE><<<grid, kPmLanes << 2, 0, st>>>(A, B, lg, lg2); break;
    case 6: k_pm_pass<3, 3, MODE><<<grid, kPmLanes << 3, 0, st>>>(A, B, lg, lg2); break;
    case 7: k_pm_pass<4, 3, MODE><<<grid, kPmLanes << 3, 0, st>>>(A, B, lg, lg2); break;
    default: k_pm_pass<4, 4, MODE><<<grid, kPmLanes << 4, 0, st>>>(A, B, lg, lg2); break;
    }
    FF_CUDA(cudaGetLastError());
    return FFSPMV_OK;
}

template <int NPR>
ffspmv_status pm_out(int ln, const u32 *Ch, u32 *C, int ne, int lg, int lg2, long long klo, long long khi, const PmOut &c,
                     cudaStream_t st)
{
    const unsigned tiles = (unsigned)((((long long)ne << (lg - ln)) + kPmLanes - 1) / kPmLanes);
    switch (ln) {
    case 4: k_pm_out<2, 2, NPR><<<tiles, kPmLanes << 2, 0, st>>>(Ch, C, ne, lg, lg2, klo, khi, c); break;
    case 5: k_pm_out<3, 2, NPR><<<tiles, kPmLanes << 2, 0, st>>>(Ch, C, ne, lg, lg2, klo, khi, c); break;
    case 6: k_pm_out<3, 3, NPR><<<tiles, kPmLanes << 3, 0, st>>>(Ch, C, ne, lg, lg2, klo, khi, c); break;
    case 7: k_pm_out<4, 3, NPR><<<tiles, kPmLanes << 3, 0, st>>>(Ch, C, ne, lg, lg2, klo, khi, c); break;
    default: k_pm_out<4, 4, NPR><<<tiles, kPmLanes << 4, 0, st>>>(Ch, C, ne, lg, lg2, klo, khi, c); break;
    }
    FF_CUDA(cudaGetLastError());
    return FFSPMV_OK;
}

// Primes whose product exceeds every exact coefficient; 0 when three do not.
int pm_primes(u32 p, int si, long long terms)
{
    const long double bound = (long double)si * (long double)terms * (long double)(p - 1) * (long double)(p - 1);
    long double prod = 1;
    for (int q = 0; q < kPmPrimes; ++q) {
        prod *= kPmP[q];
        if (bound < prod) return q + 1;
    }
    return 0;
}

// Smallest transform whose cyclic wrap leaves the coefficients klo..khi
// alone: coefficient k of the product lands on k mod L, so L > khi and
// da + db - L < klo.
int pm_length_log(long long da, long long db, long long klo, long long khi)
{
    return pm_log2(std::max(khi + 1, da + db - klo + 1));
}

// ---------------------------------------------------------------------------
// Products by the definition.  A CTA forms up to 16 x 16 or 8 x 32 entries of
// one coefficient of C (2 x 4 per lane); its eight warps take every eighth
// pair (A_a, B_(k-a)) into shared memory of their own, and their reduced sums
// meet at the end.  One launch, where the transforms need three to five: what
// short operands (the lower levels of the sigma-basis recursion) pay for.
// PD_FOLD: more terms than 64 bits hold.  PD_HALF (p <= 2^16, si and sc
// multiples of 4): two rows k, k + 1 of A in one word as they go into shared
// memory, those of B with their low bytes first, and two dot products of pairs
// (dp2a) in place of two 64-bit multiply-adds, which take twice as long; sums
// of a pair's low and high bytes are joined after each coefficient.  32 x 32
// matrices of order 100 by 100: 31 us with 64-bit multiply-adds, 23 so.
constexpr int kPdWarps = 8;
constexpr int kPdTile = 32 * 36 + 32 * 8;   // words of a warp's tiles: rows of A (padded by 4 words), then B
static_assert(16 * 36 + 32 * 16 <= kPdTile && 8 * 36 + 32 * 32 <= kPdTile, "16 rows by 16 columns, 8 rows by 32");

struct PmDirect {
    const u32 *A, *B;
    u32 *C;
    int sr, si, sc, da, db, klo;
    int si4, ast, ntj, lgn;   // si rounded up to 4, row stride of the A tile, column threads and their log2
    const int *ea, *eb;
    Mod M;
    PmNode node;
};

enum { PD_PLAIN, PD_FOLD, PD_HALF };

template <int MODE>
__global__ void __launch_bounds__(kPdWarps * 32) k_pm_direct(const __grid_constant__ PmDirect a)
{
    __shared__ __align__(16) u32 tile[kPdWarps][kPdTile];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = a.klo + blockIdx.x;
    const int da = a.ea ? min(a.da, __ldg(a.ea)) : a.da, db = a.eb ? min(a.db, __ldg(a.eb)) : a.db;
    const int nti = 32 >> a.lgn, rows = min(2 * nti, 32), i0 = blockIdx.y * rows;
    const int ti = lane >> a.lgn, tj = lane & (a.ntj - 1);
    const int cols4 = 4 * a.ntj, nr = min(rows, a.sr - i0);
    u32 *As = tile[warp], *Bs = As + rows * a.ast;
    if (nr < rows || a.si != a.si4 || a.sc != cols4) {
        // padding rows and columns are never loaded and read as zero
        for (int i = lane; i < kPdTile; i += 32) As[i] = 0u;
    }
    u64 acc[2][4];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0;
    const bool vec = (a.si & 3) == 0 && (a.sc & 3) == 0;   // rows of 16-byte blocks (device arrays are 16-byte aligned)
    const u32 *ap = As + min(ti, rows - 1) * a.ast, *ap1 = As + min(ti + nti, rows - 1) * a.ast, *bp = Bs + 4 * tj;
    for (int x = max(0, k - db) + warp; x <= min(da, k); x += kPdWarps) {
        const u32 *ag = a.A + ((size_t)x * a.sr + i0) * a.si, *bg = a.B + (size_t)(k - x) * a.si * a.sc;
        __syncwarp();
        if (MODE == PD_HALF) {
            const int qa = a.si >> 2, qb = a.sc >> 2;
            for (int e = lane; e < nr * qa; e += 32) {
                const int r = e / qa, c = e - r * qa;
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(ag) + e);
                *reinterpret_cast<uint2 *>(As + r * a.ast + 2 * c) = make_uint2(v.x | v.y << 16, v.z | v.w << 16);
            }
            for (int e = lane; e < (a.si >> 1) * qb; e += 32) {
                const int r = e / qb, c = e - r * qb;   // rows 2 r and 2 r + 1
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(bg) + 2 * r * qb + c);
                const uint4 w = __ldg(reinterpret_cast<const uint4 *>(bg) + (2 * r + 1) * qb + c);
                *reinterpret_cast<uint4 *>(Bs + r * cols4 + 4 * c) =
                    make_uint4(__byte_perm(v.x, w.x, 0x5140), __byte_perm(v.y, w.y, 0x5140), __byte_perm(v.z, w.z, 0x5140),
                               __byte_perm(v.w, w.w, 0x5140));
            }
        } else if (vec) {
            const int qa = a.si >> 2, qb = a.sc >> 2;
            for (int e = lane; e < nr * qa; e += 32) {
                const int r = e / qa, c = e - r * qa;
                *reinterpret_cast<uint4 *>(As + r * a.ast + 4 * c) = __ldg(reinterpret_cast<const uint4 *>(ag) + e);
            }
            for (int e = lane; e < a.si * qb; e += 32) {
                const int r = e / qb, c = e - r * qb;
                *reinterpret_cast<uint4 *>(Bs + r * cols4 + 4 * c) = __ldg(reinterpret_cast<const uint4 *>(bg) + e);
            }
        } else {
            for (int e = lane; e < nr * a.si; e += 32) {
                const int r = e / a.si, c = e - r * a.si;
                As[r * a.ast + c] = __ldg(ag + e);
            }
            for (int e = lane; e < a.si * a.sc; e += 32) {
                const int r = e / a.sc, c = e - r * a.sc;
                Bs[r * cols4 + c] = __ldg(bg + e);
            }
        }
        __syncwarp();
        if constexpr (MODE == PD_HALF) {
            // at most 32 products below 2^24 per sum
            u32 lo[2][4] = {}, hi[2][4] = {};
            for (int kk = 0; kk < a.si4 / 2; kk += 2) {
                const uint2 av[2] = {*reinterpret_cast<const uint2 *>(ap + kk), *reinterpret_cast<const uint2 *>(ap1 + kk)};
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const uint4 b = *reinterpret_cast<const uint4 *>(bp + (kk + u) * cols4);
                    const u32 bc[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            lo[r][c] = __dp2a_lo(u ? av[r].y : av[r].x, bc[c], lo[r][c]);
                            hi[r][c] = __dp2a_hi(u ? av[r].y : av[r].x, bc[c], hi[r][c]);
                        }
                }
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] += (u64)hi[r][c] * 256u + lo[r][c];
        }
        for (int kk = 0; MODE != PD_HALF && kk < a.si4; kk += 4) {
            const uint4 av[2] = {*reinterpret_cast<const uint4 *>(ap + kk), *reinterpret_cast<const uint4 *>(ap1 + kk)};
            uint4 bv[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) bv[r] = *reinterpret_cast<const uint4 *>(bp + (kk + r) * cols4);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const u32 ar[4] = {av[r].x, av[r].y, av[r].z, av[r].w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    acc[r][0] += (u64)ar[u] * bv[u].x;
                    acc[r][1] += (u64)ar[u] * bv[u].y;
                    acc[r][2] += (u64)ar[u] * bv[u].z;
                    acc[r][3] += (u64)ar[u] * bv[u].w;
                    if (MODE == PD_FOLD && (u & 1)) {
                        // two products below p^2 < 2^62 on top of less than p 2^32
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const u32 hi = (u32)(acc[r][c] >> 32);
                            acc[r][c] = (u64)min(hi, hi - a.M.m) << 32 | (u32)acc[r][c];
                        }
                    }
                }
            }
        }
    }
    // the warps' sums, each below p: entry (ti + nti r, 4 tj + c) at [r][c][lane]
    __syncthreads();
    u32 *red = tile[0];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) red[(warp * 8 + r * 4 + c) * 32 + lane] = red64(acc[r][c], a.M);
    __syncthreads();
    u32 *cg = a.C + (size_t)blockIdx.x * a.sr * a.sc;
    {
        const int l = lane, rc = warp;   // 256 threads: one entry each
        const int i = (l >> a.lgn) + (rc >> 2) * nti, j = 4 * (l & (a.ntj - 1)) + (rc & 3);
        u64 s = 0;
#pragma unroll
        for (int w = 0; w < kPdWarps; ++w) s += red[(w * 8 + rc) * 32 + l];
        if (i < nr && j < a.sc) cg[(size_t)(i0 + i) * a.sc + j] = red64(s, a.M);
    }
    if (a.node.out && blockIdx.x == 0 && blockIdx.y == 0 && warp == 0) pm_node(a.node, lane);
}

}  // namespace

size_t pm_product_bytes(int sr, int si, int sc, long long da, long long db, long long klo, long long khi, int npr)
{
    const int lg = pm_length_log(da, db, klo, khi);
    if (lg > kPmMaxLog) return 0;
    return ((size_t)npr * ((size_t)sr * si + (size_t)si * sc + (size_t)sr * sc) << lg) * 4;
}

ffspmv_status pm_direct(u32 p, int sr, int si, int sc, int da, int db, const u32 *A, const u32 *B, u32 *C, int klo,
                        int khi, const int *ea, const int *eb, const PmNode *node, cudaStream_t st)
{
    PmDirect a;
    memset(&a, 0, sizeof(a));
    a.A = A;
    a.B = B;
    a.C = C;
    a.sr = sr;
    a.si = si;
    a.sc = sc;
    a.da = da;
    a.db = db;
    a.klo = klo;
    a.si4 = (si + 3) / 4 * 4;
    a.ast = a.si4 + 4;
    while ((4 << a.lgn) < sc) ++a.lgn;
    a.ntj = 1 << a.lgn;
    a.ea = ea;
    a.eb = eb;
    a.M = make_mod(p, 1, 0);
    if (node) a.node = *node;
    const int rows = std::min(2 * (32 >> a.lgn), 32);
    const dim3 grid((unsigned)(khi - klo + 1), (unsigned)((sr + rows - 1) / rows));
    // terms of one warp's sum
    const unsigned __int128 terms = (unsigned __int128)si * ((std::min(da, db) + kPdWarps) / kPdWarps + 1);
    const bool fold = terms * (p - 1) * (p - 1) >= ((unsigned __int128)1 << 64);
    if (p <= 65536u && si % 4 == 0 && sc % 4 == 0) k_pm_direct<PD_HALF><<<grid, kPdWarps * 32, 0, st>>>(a);
    else if (fold) k_pm_direct<PD_FOLD><<<grid, kPdWarps * 32, 0, st>>>(a);
    else k_pm_direct<PD_PLAIN><<<grid, kPdWarps * 32, 0, st>>>(a);
    FF_CUDA(cudaGetLastError());
    return FFSPMV_OK;
}

ffspmv_status pm_product(u32 p, int sr, int si, int sc, long long da, long long db, const u32 *A_, const u32 *B_, u32 *C_,
                         long long klo, long long khi, void *work, size_t work_bytes, cudaStream_t st)
{
    // the exact coefficients must stay below the product of the primes
    const int npr = pm_primes(p, si, std::min(da, db) + 1);
    const size_t need = pm_product_bytes(sr, si, sc, da, db, klo, khi, npr);
    if (!npr || !need) return FFSPMV_ERR_UNSUPPORTED;
    if (work_bytes < need) return FFSPMV_ERR_ARG;
    ffspmv_status r;
    const int lg = pm_length_log(da, db, klo, khi);
    // L <= 256 in one pass, else two axes of at most 256 points
    const int lg2 = lg <= 8 ? 0 : lg / 2, lg1 = lg - lg2;
    const long long L = 1LL << lg;
    const int ea = sr * si, eb = si * sc, ec = sr * sc;
    u32 *Ah = (u32 *)work, *Bh = Ah + (size_t)npr * L * ea, *Ch = Bh + (size_t)npr * L * eb;
    auto tiles = [&](int ne, int ln) { return (unsigned)((((long long)ne << (lg - ln)) + kPmLanes - 1) / kPmLanes); };
    PmOp A = {A_, (da + 1) * ea, Ah, ea, tiles(ea, lg1)}, B = {B_, (db + 1) * eb, Bh, eb, tiles(eb, lg1)};
    if (lg2 == 0) {
        if ((r = pm_pass<PM_F>(lg1, A, B, lg, lg2, npr, st)) != FFSPMV_OK) return r;
    } else {
        if ((r = pm_pass<PM_F1>(lg1, A, B, lg, lg2, npr, st)) != FFSPMV_OK) return r;
        A.tiles = tiles(ea, lg2);
        B.tiles = tiles(eb, lg2);
        if ((r = pm_pass<PM_F2>(lg2, A, B, lg, lg2, npr, st)) != FFSPMV_OK) return r;
    }
    PmPw w;
    memset(&w, 0, sizeof(w));
    w.sr = sr;
    w.si = si;
    w.sc = sc;
    w.si4 = (w.si + 3) / 4 * 4;
    w.sc4 = (w.sc + 3) / 4 * 4;
    w.nti = (w.sr + 3) / 4;
    w.ntj = w.sc4 / 4;
    w.tp = kPwThreads / (w.nti * w.ntj);
    w.ast = 4 * w.nti * w.si4 + 4;   // 4 words of padding: neighbouring points start in other banks
    w.bst = w.si4 * w.sc4 + 4;
    // both matrices of every point in at most 96 KB (two CTAs per SM)
    w.tp = std::max(1, std::min(w.tp, (int)(96 * 1024 / 4) / (w.ast + w.bst)));
    w.L = (int)L;
    auto magic = [](int d) { return (u32)((((u64)1 << 32) + d - 1) / d); };
    w.m_a = magic(ea);
    w.m_si = magic(w.si);
    w.m_b = magic(eb);
    w.m_sc = magic(w.sc);
    const size_t pw_smem = (size_t)w.tp * (w.ast + w.bst) * 4;
    FF_CUDA(cudaFuncSetAttribute(k_pm_pointwise, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
    k_pm_pointwise<<<dim3((unsigned)((L + w.tp - 1) / w.tp), (unsigned)npr), kPwThreads, pw_smem, st>>>(Ah, Bh, Ch, w);
    FF_CUDA(cudaGetLastError());
    PmOut c;
    memset(&c, 0, sizeof(c));
    c.mp = make_mod(p, 1, 0);
    for (int q = 0; q < npr; ++q) {
        const u64 P = kPmP[q];
        // the pointwise products carry 2^-32, the inverse transform a factor L
        c.linv[q] = (u32)((u64)pm_pow((u64)L, P - 2, P) * (((u64)1 << 32) % P) % P);
        c.linv_q[q] = (u32)(((u64)c.linv[q] << 32) / P);
    }
    auto inv = [](u64 a, u64 P, u32 &v, u32 &vq) {
        v = pm_pow(a, P - 2, P);
        vq = (u32)(((u64)v << 32) / P);
    };
    inv(kPmP[0], kPmP[1], c.inv01, c.inv01q);
    inv(kPmP[0], kPmP[2], c.inv02, c.inv02q);
    inv(kPmP[1], kPmP[2], c.inv12, c.inv12q);
    c.p0_mod_p = (u32)(kPmP[0] % p);
    c.p0p1_mod_p = (u32)((unsigned __int128)kPmP[0] * kPmP[1] % p);
    if (lg2) {
        const PmOp Cc = {nullptr, 0, Ch, ec, tiles(ec, lg2)}, none = {nullptr, 0, nullptr, 1, 0};
        if ((r = pm_pass<PM_I1>(lg2, Cc, none, lg, lg2, npr, st)) != FFSPMV_OK) return r;
    }
    return npr == 1   ? pm_out<1>(lg1, Ch, C_, ec, lg, lg2, klo, khi, c, st)
           : npr == 2 ? pm_out<2>(lg1, Ch, C_, ec, lg, lg2, klo, khi, c, st)
                      : pm_out<3>(lg1, Ch, C_, ec, lg, lg2, klo, khi, c, st);
}

}  // namespace ff

using namespace ff;

extern "C" ffspmv_status polymat_mul_workspace(int32_t s, int64_t da, int64_t db, int64_t *bytes)
{
    if (!bytes || s < 1 || s > 32 || da < 0 || db < 0) return FFSPMV_ERR_ARG;
    if (da + db + 1 > (1LL << kPmMaxLog)) return FFSPMV_ERR_UNSUPPORTED;
    const long long L = 1LL << pm_log2(da + db + 1);
    // the planes for any p (three primes); the rest is no longer used, but callers know the size
    *bytes = 3LL * kPmPrimes * s * s * L * 4 + (long long)kPmPrimes * L * 8 + 256;
    return FFSPMV_OK;
}

extern "C" ffspmv_status polymat_mul(uint32_t p, int32_t s, int64_t da, int64_t db, const uint32_t *d_A,
                                     const uint32_t *d_B, uint32_t *d_C, void *d_work, int64_t work_bytes,
                                     ffspmv_stream_t stream)
{
    if (p < 2 || p > (1u << 31) || s < 1 || s > 32 || da < 0 || db < 0 || !d_A || !d_B || !d_C || !d_work)
        return FFSPMV_ERR_ARG;
    int64_t need = 0;
    const ffspmv_status r = polymat_mul_workspace(s, da, db, &need);
    if (r != FFSPMV_OK) return r;
    if (work_bytes < need || ((uintptr_t)d_work & 15)) return FFSPMV_ERR_ARG;
    return pm_product(p, s, s, s, da, db, d_A, d_B, d_C, 0, da + db, d_work, (size_t)work_bytes, (cudaStream_t)stream);
}
