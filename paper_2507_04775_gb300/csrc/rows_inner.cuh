// The forward row pass of ModUp's converted limbs, the key inner product and,
// on the special limbs, the inverse row pass that begins ModDown, in one
// kernel (Sec. III-F5 "Dot product fusion" taken one step further in both
// directions).
//
// A CTA owns one tile of 1024 consecutive words of one extended limb (whole
// rows).  It transforms the tile of every digit
// -- two digits at a time, which share each twiddle -- into shared memory, then
// multiplies and accumulates all digits with the two key components (128-bit
// sums, one reduction), reading the keys coalesced.  The sums of a q-limb go
// out; those of a special limb go back to shared memory and through the
// inverse row pass, so the accumulators of special limbs never leave the chip,
// nor do the transformed digits.
//
// What it replaces at logN = 16, 30 limbs, three digits: the row pass of 90
// limbs (33 us by itself), the inner product (HBM bound on 189 MB, of which 47 MB
// are the digits re-read, 37 us) and the inverse row pass of 20 limbs (13 us).
// It takes 74 us, bound by the latency of its own chain at 22 warps per SM (45 %
// of issue slots), and two launches fewer; the key words of a tile are on their
// way to L2 while the digits transform.  HMult at logN = 16: 10 limbs 106.6 ->
// 98.5 us, 17: 144.8 -> 139.4, 30: 235.0 -> 233.0; logN = 17, 36 limbs, four
// digits: 652.9 -> 627.7.  Six CTAs per SM up to three digits, five above: more
// lose to the L1 their tiles take (four digits: 197 us with five, 207 with six,
// 243 with seven).
#pragma once

#include "fides_internal.cuh"
#include "ntt.cuh"

// ---------------------------------------------------------------------------
// Operands of the key inner product (k_inner and k_rows_inner).
// ---------------------------------------------------------------------------
struct IPOp {
    const u64 *ext;     // [beta][ne][N]
    const u64 *dsrc;    // [nl][N] evaluation-form input
    const u64 *evk;     // [dnum][2][L+K][N]
    u64 *acc;           // [2][ne][N]
    int nl, ne, beta, alpha;
    u64 g;              // 0, or the Galois element through which the digits are read (hoisted rotation)
    // k_rows_inner:
    u64 *pc;            // [2][K][N]  the special limbs' sums after the inverse row pass
    u64 *xdst;          // [2][N]  the same for q-limb xl (not stored to acc), or null
    int xl;
};

// One op inline (dop == nullptr; grid.y = its ne limbs) or a device table of
// ops with a row table: row r (grid.y) computes limb drow[r] & 127 of op
// drow[r] >> 7 (an op has at most FIDES_MAX_PRIMES limbs).  The batched path orders the rows by key and key limb, so
// that the ops sharing a key (every HMult of a batch shares the
// relinearisation key) read each key limb while it is in L2.
struct IPArgs {
    const IPOp *dop;
    const int *drow;
    int nop;
    IPOp one;
};

namespace {

__device__ __forceinline__ u64 reduce_acc(const Acc128 &c, const PrimeInfo &p)
{
    return reduce128(((u64)c.w3 << 32) | c.w2, ((u64)c.w1 << 32) | c.w0, p);
}

// the same for a sum of at most two products of canonical residues
__device__ __forceinline__ u64 reduce_acc2(const Acc128 &c, const PrimeInfo &p)
{
    return csub(csub(reduce_prod(((u64)c.w3 << 32) | c.w2, ((u64)c.w1 << 32) | c.w0, p), p.q2), p.q);
}

// The same for a sum of m products of canonical residues: the Barrett form
// where its bound holds, m q^2 < 2^(k+63) for m at most 2^(63-k) (k the bit
// length of q: m <= 4 at 61-bit primes, 8 at 60-bit), reduce128 otherwise.
__device__ __forceinline__ bool reduce_prod_ok(int m, const PrimeInfo &p)
{
    return (u64)m <= (1ull << (__clzll((long long)p.q) - 1));   // 2^(63-k), k = 64 - clz(q)
}
__device__ __forceinline__ u64 reduce_accm(const Acc128 &c, const PrimeInfo &p, bool barrett)
{
    const u64 hi = ((u64)c.w3 << 32) | c.w2, lo = ((u64)c.w1 << 32) | c.w0;
    return barrett ? csub(csub(reduce_prod(hi, lo, p), p.q2), p.q) : reduce128(hi, lo, p);
}
// The same in [0, 2q).
__device__ __forceinline__ u64 reduce_accl(const Acc128 &c, const PrimeInfo &p, bool barrett)
{
    const u64 hi = ((u64)c.w3 << 32) | c.w2, lo = ((u64)c.w1 << 32) | c.w0;
    return barrett ? csub(reduce_prod(hi, lo, p), p.q2) : reduce128(hi, lo, p);
}

constexpr int RI_LE = 3;                      // elements per thread: 8

// shared memory of a CTA: one padded tile per digit, and at least the two
// accumulators
inline size_t rows_inner_smem(int max_beta)
{
    return sizeof(u64) * (1024 + 64) * (size_t)(max_beta < 2 ? 2 : max_beta);
}

// Whether key switches of up to `beta` digits over `limbs` extended limbs in all
// take the fused kernel: two-pass transforms with folding primes (digits below
// 2q: the cross products of five sum below 5 x 3 x 2^60 < 2^64), and one digit, or
// 11 limbs of logN = 16 or more.  Below, a CTA's chain of digits is longer than
// the launches it saves: HMult at logN = 14 with 7 + 3 limbs, three digits, 42.2
// -> 46.3 us, at logN = 15 with 14 + 7, two digits, 82.9 -> 85.2, with 7 + 7, one
// digit, 59.9 -> 53.7, with 20 + 10 97.4 -> 94.9; at logN = 16 with 1 + 10 limbs
// 60.5 -> 57.6, 17 + 10 145.9 -> 141.5.
inline bool rows_inner_ok(const fides_ctx *c, int beta, int limbs)
{
    return c->fold && c->logN > 12 && beta <= 5 && (beta == 1 || ((long)limbs << c->logN) >= (11L << 16));
}

// Index maps of a tile: C rows of 2^S elements, padded by a word in sixteen.
template <int S, int C>
struct RiTile {
    static constexpr int E = 1 << RI_LE;
    static constexpr int THREADS = (C << S) >> RI_LE;
    static constexpr int RT = (1 << S) >> RI_LE;
    static constexpr int R = (S + RI_LE - 1) / RI_LE;
    static constexpr int RP = (1 << S) + (1 << (S - 4));
    static __device__ __forceinline__ int w(int c, int k) { return c * RP + k + (k >> 4); }
};

// Forward rows of ND digits: src[d] is the tile of a digit in global memory,
// sm[d] receives its transform in [0, 2q).
template <int ND, int LOGN, int S, int C>
__device__ __forceinline__ void ri_forward(const u64 *const (&src)[ND], u64 *const (&sm)[ND],
                                           const TwPair *__restrict__ tw, const PrimeInfo &pr, int c, int u)
{
    using T = RiTile<S, C>;
    const FoldP fp(pr, false);
    constexpr int S0 = LOGN - S;
    const TwPair none = {0, 0};
    u64 x[ND][T::E];
#pragma unroll
    for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int r = 0; r < T::E; ++r) x[d][r] = src[d][(c << S) + kmap<RI_LE>(u, r, S - RI_LE)];
    auto Xof = [&](int b) -> int { return (((int)blockIdx.x * C + c) << (S - RI_LE - b)) | (u >> b); };
#define FIDES_RI_ROUND(RHO)                                                                          \
    if (RHO < T::R) {                                                                                \
        constexpr int b = round_window<RI_LE, S, false>(RHO < T::R ? RHO : 0);                      \
        if (RHO > 0) {                                                                               \
            _Pragma("unroll") for (int d = 0; d < ND; ++d)                                           \
                _Pragma("unroll") for (int r = 0; r < T::E; ++r)                                     \
                    x[d][r] = sm[d][T::w(c, kmap<RI_LE>(u, r, b))];                                  \
        }                                                                                            \
        ntt_round<LOGN, ND, RI_LE, false, S0, S, b, round_first<RI_LE, S>(RHO < T::R ? RHO : 0), false, false, \
                  true, false>(x, Xof(b), tw, nullptr, pr.q, pr.q2, fp, none, none);                 \
        if (RHO == T::R - 1) {                                                                       \
            _Pragma("unroll") for (int d = 0; d < ND; ++d)                                           \
                _Pragma("unroll") for (int r = 0; r < T::E; ++r) x[d][r] = fold_2q(x[d][r], fp);     \
        }                                                                                            \
        _Pragma("unroll") for (int d = 0; d < ND; ++d)                                               \
            _Pragma("unroll") for (int r = 0; r < T::E; ++r)                                         \
                sm[d][T::w(c, kmap<RI_LE>(u, r, b))] = x[d][r];                                      \
        if (RHO < T::R - 1) __syncthreads();                                                         \
    }
    FIDES_RI_ROUND(0)
    FIDES_RI_ROUND(1)
    FIDES_RI_ROUND(2)
    FIDES_RI_ROUND(3)
#undef FIDES_RI_ROUND
}

// Inverse rows of the two accumulators, from shared memory to dst[t].
template <int LOGN, int S, int C>
__device__ __forceinline__ void ri_inverse(u64 *const (&sm)[2], u64 *const (&dst)[2], const TwPair *__restrict__ tw,
                                           const PrimeInfo &pr, int c, int u)
{
    using T = RiTile<S, C>;
    const FoldP fp(pr, true);
    constexpr int S0 = LOGN - S;
    const TwPair none = {0, 0};
    u64 x[2][T::E];
    auto Xof = [&](int b) -> int { return (((int)blockIdx.x * C + c) << (S - RI_LE - b)) | (u >> b); };
#define FIDES_RI_ROUND(RHO)                                                                          \
    if (RHO < T::R) {                                                                                \
        constexpr int b = round_window<RI_LE, S, true>(RHO < T::R ? RHO : 0);                       \
        _Pragma("unroll") for (int t = 0; t < 2; ++t)                                                \
            _Pragma("unroll") for (int r = 0; r < T::E; ++r)                                         \
                x[t][r] = sm[t][T::w(c, kmap<RI_LE>(u, r, b))];                                      \
        ntt_round<LOGN, 2, RI_LE, true, S0, S, b, round_first<RI_LE, S>(RHO < T::R ? RHO : 0), false, false, \
                  true, false>(x, Xof(b), tw, nullptr, pr.q, pr.q2, fp, none, none);                 \
        if (RHO < T::R - 1) {                                                                        \
            _Pragma("unroll") for (int t = 0; t < 2; ++t)                                            \
                _Pragma("unroll") for (int r = 0; r < T::E; ++r)                                     \
                    sm[t][T::w(c, kmap<RI_LE>(u, r, b))] = x[t][r];                                  \
            __syncthreads();                                                                         \
        }                                                                                            \
    }
    FIDES_RI_ROUND(0)
    FIDES_RI_ROUND(1)
    FIDES_RI_ROUND(2)
    FIDES_RI_ROUND(3)
#undef FIDES_RI_ROUND
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int r = 0; r < T::E; ++r)
            dst[t][(c << S) + kmap<RI_LE>(u, r, S - RI_LE)] = x[t][r];
}

// Tiles of C rows of 2^S elements.  Inline op: grid.y covers the special limbs
// first (they have the most work), then the q-limbs from the last.
template <int LOGN, int S, int C, int MAXB>
__global__ void __launch_bounds__((C << S) >> RI_LE, MAXB <= 3 ? 6 : 5)
    k_rows_inner(IPArgs A, int L, int K, const PrimeInfo *__restrict__ P, const TwPair *__restrict__ TW,
                 const TwPair *__restrict__ ITW)
{
    using T = RiTile<S, C>;
    extern __shared__ u64 rsm[];
    constexpr int TILE = C * T::RP;
    const int N = 1 << LOGN, nfull = L + K;
    IPOp op;
    int z;
    if (A.dop) {
        const int r = __ldg(A.drow + blockIdx.y);
        op = A.dop[r >> 7];
        z = r & 127;
    } else {
        op = A.one;
        z = (int)blockIdx.y < K ? op.nl + (int)blockIdx.y : op.ne - 1 - (int)blockIdx.y;
    }
    const int nl = op.nl, ne = op.ne, beta = op.beta;
    const int pz = z < nl ? z : L + (z - nl);
    const int own = z < nl ? z / op.alpha : beta;
    const PrimeInfo pr = P[pz];
    const int t = threadIdx.x;
    const int c = t / T::RT, u = t % T::RT;
    u64 *tiles = rsm;
    const TwPair *__restrict__ ftw = TW + ((size_t)pz << LOGN), *__restrict__ itw = ITW + ((size_t)pz << LOGN);
    const size_t tile0 = (size_t)blockIdx.x * (C << S);
    const u64 *ext = op.ext + (size_t)z * N + tile0;
    const size_t dstep = (size_t)ne * N;
    const u64 *__restrict__ k0 = op.evk + (size_t)pz * N + tile0;
    const u64 *__restrict__ k1 = k0 + (size_t)nfull * N;
    const size_t kstep = 2 * (size_t)nfull * N;
    // the key words of this tile on their way to L2 (keys are final when
    // registered, so this may run ahead of the previous kernel)
    if (t < 2 * beta && (((uintptr_t)op.evk) & 15) == 0) {
        const u64 *k = k0 + (size_t)t * nfull * N;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(k), "r"((u32)((C << S) * 8)) : "memory");
    }
    pdl_wait();

    const bool bar = reduce_prod_ok(2 * beta, pr);
    const bool inv = z >= nl || (op.xdst && z == op.xl);   // the sums go through the inverse row pass

    // the digits that were converted to this limb's prime (all but its own)
    const int nd = beta - (own < beta ? 1 : 0);
#pragma unroll 1
    for (int m = 0; m < nd; m += 2) {
        // (opaque, so that the twiddle loads are not hoisted out of the loop
        // into registers there are not)
        const TwPair *twm = ftw;
        asm volatile("" : "+l"(twm));
        const int j0 = m + (m >= own ? 1 : 0), j1 = m + 1 + (m + 1 >= own ? 1 : 0);
        if (m + 1 < nd) {
            const u64 *const src[2] = {ext + j0 * dstep, ext + j1 * dstep};
            u64 *const sm[2] = {tiles + j0 * TILE, tiles + j1 * TILE};
            ri_forward<2, LOGN, S, C>(src, sm, twm, pr, c, u);
        } else {
            const u64 *const src[1] = {ext + j0 * dstep};
            u64 *const sm[1] = {tiles + j0 * TILE};
            ri_forward<1, LOGN, S, C>(src, sm, twm, pr, c, u);
        }
    }
    __syncthreads();

    // inner product
    const u64 *dsrc = op.dsrc + (size_t)z * N + tile0;
    u64 *acc = op.acc + (size_t)z * N + tile0;
    // UN elements at a time, every load issued before the first product
    constexpr int UN = MAXB <= 4 ? 2 : 1;
#pragma unroll 1
    for (int i = 0; i < T::E; i += UN) {
        u64 x[UN][MAXB], y0[UN][MAXB], y1[UN][MAXB];
#pragma unroll
        for (int v = 0; v < UN; ++v) {
            const int e = t + T::THREADS * (i + v);
#pragma unroll
            for (int j = 0; j < MAXB; ++j)
                if (j < beta) {
                    y0[v][j] = k0[j * kstep + e];
                    y1[v][j] = k1[j * kstep + e];
                }
        }
#pragma unroll
        for (int v = 0; v < UN; ++v) {
            const int e = t + T::THREADS * (i + v);
            const int w = T::w(e >> S, e & ((1 << S) - 1));
#pragma unroll
            for (int j = 0; j < MAXB; ++j)
                if (j < beta) x[v][j] = j == own ? dsrc[e] : tiles[j * TILE + w];
        }
#pragma unroll
        for (int v = 0; v < UN; ++v) {
            const int e = t + T::THREADS * (i + v);
            const int w = T::w(e >> S, e & ((1 << S) - 1));
            AccCols b0 = {0, 0, 0, 0}, b1 = {0, 0, 0, 0};
#pragma unroll
            for (int j = 0; j < MAXB; ++j)
                if (j < beta) {
                    mac_cols(b0, x[v][j], y0[v][j]);
                    mac_cols(b1, x[v][j], y1[v][j]);
                }
            const u64 r0 = reduce_accl(cols_sum(b0), pr, bar), r1 = reduce_accl(cols_sum(b1), pr, bar);
            if (!inv) {
                acc[e] = r0;
                acc[(size_t)ne * N + e] = r1;
            } else {
                tiles[w] = r0;              // this thread was the last reader of these words
                tiles[TILE + w] = r1;
            }
        }
    }
    if (!inv) return;
    __syncthreads();

    // the inverse row pass of both sums
    u64 *pc = (z < nl ? op.xdst : op.pc + (size_t)(z - nl) * N) + tile0;
    u64 *const sm[2] = {tiles, tiles + TILE};
    u64 *const dst[2] = {pc, pc + (z < nl ? (size_t)N : (size_t)K * N)};
    ri_inverse<LOGN, S, C>(sm, dst, itw, pr, c, u);
}

}  // namespace

// Launches k_rows_inner over `limbs` rows (one op: its extended limbs).
int ntt_rows_inner(const fides_ctx *c, const IPArgs &A, int limbs, int max_beta, cudaStream_t st);
