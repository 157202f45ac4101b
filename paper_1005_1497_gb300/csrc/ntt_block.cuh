// ntt_block.cuh -- the whole-sequence convolution by blocks: transforms that
// stop BB = 2 levels early, and short polynomial products in place of the
// pointwise product.
//
// The forward tree (ntt_core.cuh) splits x^N - 1 level by level; after
// L - BB levels it has reached the factors x^4 - c_j, c_j = +-z_i, and the
// 2^BB consecutive elements 4 j .. 4 j + 3 are the residue of the sequence
// modulo factor j.  The convolution theorem (Sec. I) holds for any such
// factorisation, so h is f g modulo each x^4 - c_j: sixteen products of two
// residues, accumulated in double words, and one Montgomery reduction per
// output.  Seen per element this is the transform of length N' = N / 4 of
// each of the four subsequences t = 4 t' + r, with the root w^4: its
// twiddles are the first N / 8 entries of the plan's table, and its inverse
// is N'^{-1} R' F' with R' the reversal of t' (Eq. 3 at length N'), so the
// output of position (t', r) belongs at index 4 <-t'>_N' + r.
//
// Why: the whole-sequence kernels are bound by the integer multiply pipe.
// Two levels of three transforms and the pointwise product took 42.9 cycles
// per element, warp and scheduler of the SM on GB300; the 4 x 4 block
// products take 30.5 (2 x 2 blocks with one level: 29.3, but half the gain
// in the table and the layout below).  The twiddle table in shared memory
// shrinks fourfold, the inverse passes' twiddle reads have 8 distinct
// addresses per warp instead of 32, and aligned groups of four elements
// stay together from input to output, so that a column/row kernel moves
// them with 8- and 16-byte accesses.  Measured on GB300 against the complete
// transform (alternating runs, bit-identical): 20011 x 2^8 39.6 -> 35.1 us,
// 4096 x 2^14 418 -> 400 us (with the staged loads that the smaller table
// makes room for: 380 us), 301 x 2^13 of 64-bit words 67.4 -> 59.4 us.
//
// Bounds (m < 2^B / 128; the static_asserts below follow them level by
// level).  Forward: inputs < m; unit butterflies at node 0 of levels 0, 1, 2,
// the others' products add 2m: below 26m for N <= 2^14 (lazy_forward).  A
// block product sums four products of such values (c_j g is a Shoup product,
// < 2m): T < 2704 m^2 < 2^(2B - 2), and Montgomery's reduction leaves T / 2^B
// + m < 23m.  Inverse: 46m and 92m after the two levels with unit
// butterflies, 2m more for each of the other ten: at most 112m, below the
// word.  The last factor 2^BB N^{-1} 2^B (Shoup) takes any word and brings
// N'^{-1} and Montgomery's 2^B.
// Roomy 64-bit moduli (r64, m < 2^48; N <= 2^13): products below 13m.  A
// twiddled node of levels 1 and 2 reaches 15m and 28m, so 132m forward; T <
// 69696 m^2 < 2^113, Montgomery's result below 3m (the 23m of the others is
// what the unit butterfly adds); 92m + 9 13m = 209m < 2^8 m < 2^56 inverse.
#pragma once

#include "ntt_core.cuh"

namespace ntt {

constexpr int BB = 2;                        // levels left out; blocks of 2^BB elements
// Lengths below 2^BLOCK_LMIN keep the complete transform (a thread then
// holds fewer than two blocks).
constexpr int BLOCK_LMIN = BB + 1;

// Bound of the inverse's `levels` levels, in multiples of m: unit butterflies
// on values below 23m and 46m at levels 0 and 1, products below P m.
__host__ __device__ constexpr int lazy_inverse(int levels, int P)
{
    int b = 23;
    for (int l = 0; l < levels; ++l) b = l < 2 && 2 * b > b + P ? 2 * b : b + P;
    return b;
}
// T / 2^B + m for four products of values below F m, m < 2^(B - room), in multiples of m (rounded up)
__host__ __device__ constexpr long long lazy_product(long long F, int room) { return ((4 * F * F) >> room) + 2; }
static_assert(lazy_forward(14 - BB, 2, 2) == 26 && lazy_product(26, 7) <= 23 && lazy_inverse(14 - BB, 2) == 112, "m < 2^B / 128, N <= 2^14");
static_assert(lazy_forward(13 - BB, 2, ROOMY_M2) == 132 && lazy_product(132, 64 - ROOMY_BITS) <= 3 && lazy_inverse(13 - BB, ROOMY_M2) == 209 &&
              209 < 1 << (56 - ROOMY_BITS), "r64, N <= 2^13");

template <typename W> struct Wide;
template <> struct Wide<uint32_t> { using T = uint64_t; };
template <> struct Wide<uint64_t> { using T = unsigned __int128; };
template <> struct Wide<r64> { using T = unsigned __int128; };

__device__ __forceinline__ uint32_t mont(uint64_t T, const ModC<uint32_t> &c)
{
    const uint32_t q = (uint32_t)T * c.mneg;
    return (uint32_t)((T + (uint64_t)q * c.m) >> 32);
}

template <typename W>
__device__ __forceinline__ W mont(unsigned __int128 T, const ModC<W> &c)
{
    const W lo = (W)T, q = lo * c.mneg;
    return (W)(T >> 64) + __umul64hi(q, c.m) + (lo != 0 ? 1 : 0);
}

// Shared-memory rows of the block form.  32-bit words with rows of at least
// 2^8: four pad words every 32, so that a thread's aligned groups of four
// are 16-byte accesses (conflict-free: eight lanes of the contiguous layout
// start 36 words apart) and the strided layouts stay conflict-free; all
// others one pad word, as in Geo.  Rows of fewer than 32 threads share a
// warp: their regions lie GS words apart, an odd multiple of T, which spreads
// a warp's groups over all banks.
template <typename W, int LR>
struct BGeo : Geo<W, LR> {
    using G = Geo<W, LR>;
    static constexpr bool VX = sizeof(W) == 4 && LR >= 8;
    static constexpr int PADW = VX ? 4 : 1;
    static constexpr int ROWP = G::ROW + PADW * (G::ROW >> G::PADSH);
    static constexpr int BANKS = (int)(128 / sizeof(W));
    static constexpr int GS = G::T < BANKS ? (2 * ROWP / G::T | 1) * G::T : 2 * ROWP;
    __host__ __device__ static constexpr uint32_t pad(uint32_t x) { return x + PADW * (x >> G::PADSH); }
};

template <typename W, int LR, int P>
__device__ __forceinline__ void bstore(const W (&v)[Geo<W, LR>::R], W *S, uint32_t tau)
{
    using G = BGeo<W, LR>;
    const uint32_t bp = G::pad(G::base(P, tau));
    if constexpr (G::VX && G::lo(P) == 0) {
#pragma unroll
        for (int k = 0; k < G::R; k += 4)
            *reinterpret_cast<uint4 *>(S + bp + k) = make_uint4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < G::R; ++k) S[bp + G::pad((uint32_t)k << G::lo(P))] = v[k];
    }
}

template <typename W, int LR, int P>
__device__ __forceinline__ void bload(W (&v)[Geo<W, LR>::R], const W *S, uint32_t tau)
{
    using G = BGeo<W, LR>;
    const uint32_t bp = G::pad(G::base(P, tau));
    if constexpr (G::VX && G::lo(P) == 0) {
#pragma unroll
        for (int k = 0; k < G::R; k += 4) {
            const uint4 q = *reinterpret_cast<const uint4 *>(S + bp + k);
            v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < G::R; ++k) v[k] = S[bp + G::pad((uint32_t)k << G::lo(P))];
    }
}

// Forward levels of pass P down to element bit BB, highest first.
template <typename W, int L, int LR, int P, int JJ, bool Z0>
__device__ __forceinline__ void bfwd_levels(W (&v)[2][Geo<W, LR>::R], uint32_t xbase, const W *__restrict__ tw,
                                            const ModC<W> &c)
{
    if constexpr (JJ >= 0 && Geo<W, LR>::lo(P) + JJ >= BB) {
        fwd_level<W, L, LR, P, JJ, 2, TW_SMEM, Z0, 2>(v, xbase, tw, c);
        bfwd_levels<W, L, LR, P, JJ - 1, Z0>(v, xbase, tw, c);
    }
}

// All forward passes of the rows at S and S + ROWP.
template <typename W, int L, int LR, int P, bool Z0>
__device__ __forceinline__ void bfwd_all(W (&v)[2][Geo<W, LR>::R], uint32_t rowoff, uint32_t tau, W *S, int gid,
                                         const W *__restrict__ tw, const ModC<W> &c)
{
    using G = BGeo<W, LR>;
    bfwd_levels<W, L, LR, P, G::nb(P) - 1, Z0>(v, rowoff + G::base(P, tau), tw, c);
    if constexpr (P + 1 < G::NPASS) {
        group_sync<G::T>(gid);
        bstore<W, LR, P>(v[0], S, tau);
        bstore<W, LR, P>(v[1], S + G::ROWP, tau);
        group_sync<G::T>(gid);
        bload<W, LR, P + 1>(v[0], S, tau);
        bload<W, LR, P + 1>(v[1], S + G::ROWP, tau);
        bfwd_all<W, L, LR, P + 1, Z0>(v, rowoff, tau, S, gid, tw, c);
    }
}

// The four elements from v[0][b] on <- their product with those from v[1][b]
// on modulo x^4 - z, or x^4 + z (plus), times 2^-B.
template <typename W, int R>
__device__ __forceinline__ void block_product(W (&v)[2][R], const int b, const bool plus, W z, W zp, const ModC<W> &c)
{
    using D = typename Wide<W>::T;
    const W f0 = v[0][b], f1 = v[0][b + 1], f2 = v[0][b + 2], f3 = v[0][b + 3];
    const W g0 = v[1][b], g1 = v[1][b + 1], g2 = v[1][b + 2], g3 = v[1][b + 3];
    W y1 = shoup<W>(g1, z, zp, c.m), y2 = shoup<W>(g2, z, zp, c.m), y3 = shoup<W>(g3, z, zp, c.m);
    if (plus) { y1 = c.m2 - y1; y2 = c.m2 - y2; y3 = c.m2 - y3; }
    v[0][b] = mont((D)f0 * g0 + (D)f1 * y3 + (D)f2 * y2 + (D)f3 * y1, c);
    v[0][b + 1] = mont((D)f0 * g1 + (D)f1 * g0 + (D)f2 * y3 + (D)f3 * y2, c);
    v[0][b + 2] = mont((D)f0 * g2 + (D)f1 * g1 + (D)f2 * g0 + (D)f3 * y3, c);
    v[0][b + 3] = mont((D)f0 * g3 + (D)f1 * g2 + (D)f2 * g1 + (D)f3 * g0, c);
}

// v[0] <- v[0] v[1] modulo the factors of the thread's R consecutive
// elements (first at index xbase): blocks 2i and 2i + 1 modulo x^4 - z_i and
// x^4 + z_i, times 2^-B.
template <typename W, int R>
__device__ __forceinline__ void block_products(W (&v)[2][R], uint32_t xbase, const W *__restrict__ tw, const ModC<W> &c)
{
    constexpr int CNT = R >> (BB + 1);
    constexpr int CH = (CNT >= 2 && tw_per_chunk<W>() == 2) ? 2 : 1;
    const uint32_t nb = xbase >> (BB + 1);
#pragma unroll
    for (int t0 = 0; t0 < CNT; t0 += CH) {
        W z[CH], zp[CH];
        load_tw<W, CH, TW_SMEM>(tw, nb, (uint32_t)t0, z, zp);
#pragma unroll
        for (int tt = 0; tt < CH; ++tt)
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                block_product<W, R>(v, ((t0 + tt) << (BB + 1)) + (s << BB), s == 1, z[tt], zp[tt], c);
            }
    }
}

// Inverse (decimation in time) level of element bit lo_P + JJ: level
// l = lo_P + JJ - BB of the length-N' transforms.  Its twiddle index is the
// reversal of the l bits of x >> BB below it: thread bits first, then
// register bits; the FR free register bits below BB share a twiddle.
template <typename W, int LR, int P, int JJ>
__device__ __forceinline__ void bdit_level(W (&v)[Geo<W, LR>::R], uint32_t xbase, const W *__restrict__ tw,
                                           const ModC<W> &c)
{
    using G = Geo<W, LR>;
    constexpr int R = G::R, lo = G::lo(P), l = lo + JJ - BB;
    constexpr int FR = lo < BB ? BB - lo : 0, TB = lo > BB ? lo - BB : 0;
    if constexpr (l == 0) {
        const W bound = 23 * c.m;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (k & (1 << JJ)) continue;
            ct_bfly_unit<W>(v[k], v[k | (1 << JJ)], bound);
        }
    } else {
        constexpr int CNT = 1 << (JJ - FR);
        constexpr int CH = (CNT >= 2 && tw_per_chunk<W>() == 2) ? 2 : 1;
        uint32_t tlo = 0;
        if constexpr (TB > 0) tlo = __brev((xbase & ((1u << lo) - 1u)) >> BB) >> (32 - TB);
        const uint32_t run = tlo << (JJ - FR);
#pragma unroll
        for (int t0 = 0; t0 < CNT; t0 += CH) {
            W z[CH], zp[CH];
            load_tw<W, CH, TW_SMEM>(tw, run, (uint32_t)t0, z, zp);
#pragma unroll
            for (int tt = 0; tt < CH; ++tt) {
                const int j = brv_c<JJ - FR>(t0 + tt) << FR;
#pragma unroll
                for (int hi = 0; hi < (R >> (JJ + 1)); ++hi)
#pragma unroll
                    for (int e = 0; e < (1 << FR); ++e) {
                        const int k = (hi << (JJ + 1)) | j | e;
                        if (TB == 0 && l == 1 && t0 + tt == 0) ct_bfly_unit<W>(v[k], v[k | (1 << JJ)], 46 * c.m);
                        else ct_bfly<W>(v[k], v[k | (1 << JJ)], z[tt], zp[tt], c);
                    }
            }
        }
    }
}

template <typename W, int LR, int P, int JJ>
__device__ __forceinline__ void bdit_levels(W (&v)[Geo<W, LR>::R], uint32_t xbase, const W *__restrict__ tw,
                                            const ModC<W> &c)
{
    if constexpr (JJ < Geo<W, LR>::nb(P)) {
        if constexpr (Geo<W, LR>::lo(P) + JJ >= BB) bdit_level<W, LR, P, JJ>(v, xbase, tw, c);
        bdit_levels<W, LR, P, JJ + 1>(v, xbase, tw, c);
    }
}

// All inverse passes of the row at S, from pass P down to pass 0.
template <typename W, int LR, int P>
__device__ __forceinline__ void bdit_all(W (&v)[Geo<W, LR>::R], uint32_t tau, W *S, int gid, const W *__restrict__ tw,
                                         const ModC<W> &c)
{
    using G = BGeo<W, LR>;
    bdit_levels<W, LR, P, 0>(v, G::base(P, tau), tw, c);
    if constexpr (P > 0) {
        group_sync<G::T>(gid);
        bstore<W, LR, P>(v, S, tau);
        group_sync<G::T>(gid);
        bload<W, LR, P - 1>(v, S, tau);
        bdit_all<W, LR, P - 1>(v, tau, S, gid, tw, c);
    }
}

// Output index of position x: 4 <-x'>_N' + r for x = 4 x' + r.
template <int L>
__device__ __forceinline__ uint32_t block_out(uint32_t x)
{
    constexpr uint32_t NP = 1u << (L - BB);
    return (((NP - (x >> BB)) & (NP - 1u)) << BB) | (x & ((1u << BB) - 1u));
}

// ---- columns of the column/row kernel, VEC adjacent columns at a time ----

// VEC consecutive words from / to p, one access when `wide` (p aligned).
template <typename W, int VEC>
__device__ __forceinline__ void ld_vec(const W *p, W (&d)[VEC], bool wide)
{
    if constexpr (VEC == 4 && sizeof(W) == 4) {
        if (wide) { const uint4 q = *reinterpret_cast<const uint4 *>(p); d[0] = q.x; d[1] = q.y; d[2] = q.z; d[3] = q.w; return; }
    } else if constexpr (VEC == 2 && sizeof(W) == 4) {
        if (wide) { const uint2 q = *reinterpret_cast<const uint2 *>(p); d[0] = q.x; d[1] = q.y; return; }
    } else if constexpr (VEC == 2) {
        if (wide) { const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(p); d[0] = q.x; d[1] = q.y; return; }
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) d[e] = p[e];
}

template <typename W, int VEC>
__device__ __forceinline__ void st_vec(W *p, const W (&d)[VEC], bool wide)
{
    if constexpr (VEC == 4 && sizeof(W) == 4) {
        if (wide) { *reinterpret_cast<uint4 *>(p) = make_uint4(d[0], d[1], d[2], d[3]); return; }
    } else if constexpr (VEC == 2 && sizeof(W) == 4) {
        if (wide) { *reinterpret_cast<uint2 *>(p) = make_uint2(d[0], d[1]); return; }
    } else if constexpr (VEC == 2) {
        if (wide) { *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(d[0], d[1]); return; }
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) p[e] = d[e];
}

// Inverse levels l = RW - BB + J of VEC adjacent columns of RC = 2^LC
// elements at v[OFF + e RC ..], which lie in one block and so share their
// twiddles: the run of tlo = brv(column >> BB).
template <typename W, int LC, int VEC, int OFF, int J, int RR>
__device__ __forceinline__ void bcold_levels(W (&v)[RR], uint32_t tlo, const W *__restrict__ tw, const ModC<W> &c)
{
    if constexpr (J < LC) {
        constexpr int RC = 1 << LC, CNT = 1 << J;
        constexpr int CH = (CNT >= 2 && tw_per_chunk<W>() == 2) ? 2 : 1;
        const uint32_t run = tlo << J;
#pragma unroll
        for (int t0 = 0; t0 < CNT; t0 += CH) {
            W z[CH], zp[CH];
            load_tw<W, CH, TW_SMEM>(tw, run, (uint32_t)t0, z, zp);
#pragma unroll
            for (int tt = 0; tt < CH; ++tt) {
                const int j = brv_c<J>(t0 + tt);
#pragma unroll
                for (int hi = 0; hi < (RC >> (J + 1)); ++hi)
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        const int k = OFF + e * RC + ((hi << (J + 1)) | j);
                        ct_bfly<W>(v[k], v[k | (1 << J)], z[tt], zp[tt], c);
                    }
            }
        }
        bcold_levels<W, LC, VEC, OFF, J + 1, RR>(v, tlo, tw, c);
    }
}

}  // namespace ntt
