// ntt_kernels.cuh -- kernels of the exact digital convolution, templated on
// the word type W (uint32_t / uint64_t) and on log2 N.
#pragma once

#include <type_traits>

#include "ntt_block.cuh"
#include "ntt_exact.cuh"

namespace ntt {

constexpr int BLOCK = 512;                 // threads of every row-kernel block (default)
// The whole-sequence fused kernels also come with BLK = 256: half the rows
// in flight and half the shared memory per block, so two blocks share an SM
// and pass through their barrier-separated phases independently; the
// autotuner picks per length (BLOCK for the longest whole length, whose
// rows need 512 threads).
constexpr int BLOCK_HALF = 256;

template <typename W> struct LRMax;        // longest row one block transforms
template <> struct LRMax<uint32_t> { static constexpr int v = 14; };
template <> struct LRMax<uint64_t> { static constexpr int v = 13; };
template <> struct LRMax<r64> { static constexpr int v = 13; };

// One convolution of an uneven batch, as seen by the device.
template <typename W> struct DevDesc {
    const W *f;
    const W *g;
    W *h;
};

// Arguments of the row kernels.  For a whole-sequence launch (L == LR) row
// rho is pair pair0 + rho of the batch: SRC 0 contiguous arrays f, g, h, SRC 1
// the descriptor list, SRC 2 contiguous arrays in page-locked host memory.  For the split path (L > LR) rho counts rows of the
// current wave inside the scratch arrays f (= F~, overwritten by H~) and g.
template <typename W> struct RowArgs {
    const W *f;
    const W *g;
    W *h;
    const DevDesc<W> *descs;
    long long nrows;
    long long pair0;
    const W *tw;
    ModC<W> c;
};

// Shared-memory copy of the twiddle table of a whole-sequence kernel (N/2 pairs).
template <typename W, int L>
struct TwBytes {
    static constexpr uint32_t pairs = L >= 1 ? (1u << (L - 1)) : 1u;
    static constexpr size_t v = ((size_t)pairs * 2 * sizeof(W) + 15) / 16 * 16;
};

template <typename W, int L, int LR, int BLK = BLOCK>
struct RowShape {
    using G = Geo<W, LR>;
    static constexpr int GPC = BLK / G::T;     // rows in flight per block
    static constexpr size_t smem(int ns) { return (size_t)GPC * ns * G::ROWP * sizeof(W); }
};

// Shared memory of the one-warp fused kernel: the twiddles (the first N / 8
// pairs for lengths that convolve by blocks) and, for lengths of more than
// one register pass, two rows per group and a plain one for the next f (the
// next g goes into g's row once the products are done with it).  Measured on
// GB300 against loading at the start of each pair: 20011 x 2^8 35.1 -> 32.2 us.
template <typename W, int L, int BLK = BLOCK>
struct FusedShape {
    static constexpr bool BLOCKS = L >= BLOCK_LMIN;
    using G = BGeo<W, L>;
    static constexpr int GPC = BLK / G::T;
    static constexpr int TWL = BLOCKS ? L - BB : L;     // TwBytes: 2^(TWL - 1) pairs
    static constexpr bool STAGE = G::NPASS > 1;         // the next pair staged by asynchronous copies
    static constexpr int GS = STAGE ? G::GS : 0;
    // words per asynchronous copy that keep every group's rows aligned
    static constexpr uint32_t CH = 16 / sizeof(W) > 2 && G::GS % 4 == 0 && G::ROWP % 4 == 0 ? 4 : G::GS % 2 == 0 && G::ROWP % 2 == 0 ? 2 : 1;
    static constexpr size_t next = TwBytes<W, TWL>::v + ((size_t)GPC * GS * sizeof(W) + 15) / 16 * 16;
    static constexpr size_t smem = next + (STAGE ? (size_t)GPC * G::ROW * sizeof(W) : 0);
};

// Hint: fetch `bytes` bytes at p into L2 with one bulk copy-engine
// request (no registers, no shared memory).  Skipped unless 16-byte aligned.
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes)
{
    if (((uintptr_t)p & 15u) == 0 && bytes >= 16)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes & ~15u) : "memory");
}

// Asynchronous copies into shared memory, and the wait for all of this
// thread's (visible to others after the next barrier).
template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// N = 2^L consecutive words by the T threads of a group, CH words per copy
// where the source allows.
template <typename W, int L, uint32_t CH>
__device__ __forceinline__ void stage_seq(const W *src, W *dst, uint32_t tau)
{
    using G = Geo<W, L>;
    if (CH > 1 && G::R % CH == 0 && ((uintptr_t)src & (CH * sizeof(W) - 1)) == 0) {
#pragma unroll
        for (uint32_t i = 0; i < G::R / CH; ++i) cp_async<CH * sizeof(W)>(dst + (tau + G::T * i) * CH, src + (tau + G::T * i) * CH);
    } else {
#pragma unroll 8
        for (uint32_t i = 0; i < G::R; ++i) cp_async<sizeof(W)>(dst + tau + G::T * i, src + tau + G::T * i);
    }
}

// Input and output of the fused bodies: plain words (the default), or the
// ends of the exact convolution fused in -- signed 64-bit inputs reduced
// modulo the launch's prime (IN64), and for the last of GARNER primes the
// Chinese remainder reconstruction of each output, written as a signed
// 64-bit integer.
struct NoExact { static constexpr bool IN64 = false; static constexpr int GARNER = 0; };
struct ExactOne { static constexpr bool IN64 = true; static constexpr int GARNER = 1; };
struct ExactLast { static constexpr bool IN64 = false; static constexpr int GARNER = 2; };

// Element i of a sequence whose first element is at base.
template <class X, typename W>
__device__ __forceinline__ W ld_elem(const W *base, uint32_t i, const ExactFused *xa, const ModC<W> &c)
{
    if constexpr (X::IN64) return (W)residue_fused(reinterpret_cast<const long long *>(base)[i], *xa, (uint32_t)c.m, (uint32_t)c.onep);
    else return base[i];
}

// Sequence `pair` of a contiguous batch of words (or of signed 64-bit words).
template <class X, typename W>
__device__ __forceinline__ const W *seq_base(const W *batch, long long pair, uint32_t N)
{
    if constexpr (X::IN64) return reinterpret_cast<const W *>(reinterpret_cast<const long long *>(batch) + (size_t)pair * N);
    else return batch + (size_t)pair * N;
}

// Canonical output r at index idx of sequence `pair` (hp: that sequence's words).
template <class X, typename W>
__device__ __forceinline__ void st_out(W *hp, long long pair, uint32_t N, uint32_t idx, W r, const ExactFused *xa, const ModC<W> &c)
{
    if constexpr (X::GARNER > 0) {
        const size_t at = (size_t)pair * N + idx;
        xa->h64[at] = garner_fused<X::GARNER>((uint32_t)r, X::GARNER == 2 ? xa->prev[at] : 0u, *xa, (uint32_t)c.m, (uint32_t)c.onep);
    } else {
        hp[idx] = r;
    }
}

// VEC consecutive 64-bit inputs reduced, and VEC consecutive outputs
// reconstructed (idx a multiple of VEC), two per access where aligned.
template <int VEC, typename W>
__device__ __forceinline__ void ld_residues(const long long *p, W (&d)[VEC], bool wide, const ExactFused *xa, const ModC<W> &c)
{
    long long x[VEC];
    if (wide && VEC > 1) {
#pragma unroll
        for (int e = 0; e < VEC; e += 2) {
            const longlong2 q = *reinterpret_cast<const longlong2 *>(p + e);
            x[e] = q.x; x[e + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < VEC; ++e) x[e] = p[e];
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) d[e] = (W)residue_fused(x[e], *xa, (uint32_t)c.m, (uint32_t)c.onep);
}

template <int K, int VEC, typename W>
__device__ __forceinline__ void st_garner(size_t at, const W (&r)[VEC], const W *r0, bool wide, const ExactFused *xa, const ModC<W> &c)
{
    long long h[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) h[e] = garner_fused<K>((uint32_t)r[e], K == 2 ? (uint32_t)r0[e] : 0u, *xa, (uint32_t)c.m, (uint32_t)c.onep);
    if (wide && VEC > 1) {
#pragma unroll
        for (int e = 0; e < VEC; e += 2) *reinterpret_cast<longlong2 *>(xa->h64 + at + e) = make_longlong2(h[e], h[e + 1]);
    } else {
#pragma unroll
        for (int e = 0; e < VEC; ++e) xa->h64[at + e] = h[e];
    }
}

// Words per access of one thread's R consecutive words: 16 bytes, or single
// words where there are fewer.
template <typename W, int R> __host__ __device__ constexpr int row_vec() { return R * sizeof(W) >= 16 ? (int)(16 / sizeof(W)) : 1; }

// R consecutive words from p, 16 bytes at a time where p allows.
template <typename W, int R>
__device__ __forceinline__ void ld_row(const W *p, W (&d)[R])
{
    constexpr int VEC = row_vec<W, R>();
    auto all = [&](bool wide) {
#pragma unroll
        for (int k = 0; k < R; k += VEC) {
            W t[VEC];
            ld_vec<W, VEC>(p + k, t, wide);
#pragma unroll
            for (int e = 0; e < VEC; ++e) d[k + e] = t[e];
        }
    };
    if (((uintptr_t)p & (VEC * sizeof(W) - 1)) == 0) all(true);
    else all(false);
}

// Fused convolution of whole sequences (L <= LR_max), persistent.  The block
// stages the twiddle table in shared memory once.  Per pair, f and g are
// transformed together (one set of twiddle reads serves both) through shared
// regions 0 and 1, multiplied block by block (ntt_block.cuh; lengths below 8
// pointwise), and sent back through region 0 by the decimation-in-time
// inverse; results are stored canonical.
// Each group brings its next pair by asynchronous copies while it convolves
// this one (lengths of one register pass and the exact inputs: loads, with the
// next pair asked into L2).
// Rows [base + group, a.nrows) by steps of stride.
template <typename W, int L, int SRC, class X = NoExact, int BLK = BLOCK>
__device__ __forceinline__ void conv_fused_body(const RowArgs<W> &a, long long base, long long stride,
                                                const ExactFused *xa = nullptr)
{
    using G = Geo<W, L>;
    using SH = FusedShape<W, L, BLK>;
    constexpr int T = G::T, R = G::R;
    constexpr uint32_t N = 1u << L;
    constexpr int last = G::NPASS - 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gid = threadIdx.x / T;
    const uint32_t tau = threadIdx.x % T;
    W *stw = reinterpret_cast<W *>(smem_raw);
    W *S = reinterpret_cast<W *>(smem_raw + TwBytes<W, SH::TWL>::v) + (size_t)gid * SH::GS;
    const uint32_t b0 = G::base(0, tau);
    constexpr int lo0 = G::lo(0);
    stage_twiddles<W>(a.tw, stw, TwBytes<W, SH::TWL>::pairs);
    __syncthreads();

    auto ptrs = [&](long long rho, const W *&fp, const W *&gp, W *&hp) {
        const long long pair = a.pair0 + rho;
        if constexpr (SRC == 1) {
            const DevDesc<W> d = a.descs[pair];
            fp = d.f; gp = d.g; hp = d.h;
        } else {
            fp = seq_base<X>(a.f, pair, N); gp = seq_base<X>(a.g, pair, N);
            hp = X::GARNER ? nullptr : a.h + (size_t)pair * N;
        }
    };
    constexpr uint32_t INB = X::IN64 ? 8u : (uint32_t)sizeof(W);     // bytes per input element
    constexpr bool STAGE = SH::STAGE && !X::IN64 && SRC != 2;
    // One thread per pair: its sequences are consecutive words, read and
    // written by 16-byte accesses.  By single words every access of a warp
    // touches 32 lines and counts on the L1 cache to bring the other words of
    // their sectors once, which the persistent launch, whose longest length
    // takes most of the SM's shared memory, leaves no room for: measured on
    // GB300, a batch plan of 1000 pairs of each of 2^0 .. 2^10 by single words
    // 77 us, by 16 bytes 40 (61 when that launch took 64 KB less), 3000 of 2^0
    // .. 2^9 of 64-bit words 85 and 76 (76); 37450 x 2^5 alone 11 us (30 for
    // the complete transform by single words).
    constexpr bool WHOLE = T == 1 && SH::BLOCKS && std::is_same<X, NoExact>::value;
    W *B = reinterpret_cast<W *>(smem_raw + SH::next) + (size_t)gid * N;
    using BG = BGeo<W, L>;
    const W *fp, *gp, *fn = nullptr, *gn = nullptr;
    W *hp, *hn = nullptr;
    if constexpr (STAGE) {
        if (base + gid < a.nrows) {
            ptrs(base + gid, fn, gn, hn);
            stage_seq<W, L, SH::CH>(fn, B, tau);
            stage_seq<W, L, SH::CH>(gn, S + BG::ROWP, tau);
            cp_async_wait();
            group_sync<T>(gid);
        }
    }
    for (long long rho = base + gid; rho < a.nrows; rho += stride) {
        const bool more = rho + stride < a.nrows;
        if constexpr (STAGE) hp = hn;
        else ptrs(rho, fp, gp, hp);
        if (more) {
            ptrs(rho + stride, fn, gn, hn);
            if (!STAGE && tau == 0) {
                prefetch_l2(fn, N * INB);
                prefetch_l2(gn, N * INB);
            }
        }
        W v[2][R];
        if constexpr (WHOLE) {
            ld_row<W, R>(fp, v[0]);
            ld_row<W, R>(gp, v[1]);
        } else {
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const uint32_t x = b0 + ((uint32_t)k << lo0);
                if constexpr (STAGE) {
                    v[0][k] = B[x];
                    v[1][k] = S[BG::ROWP + x];
                } else {
                    v[0][k] = ld_elem<X>(fp, x, xa, a.c);
                    v[1][k] = ld_elem<X>(gp, x, xa, a.c);
                }
            }
        }
        if constexpr (STAGE) {
            group_sync<T>(gid);
            if (more) stage_seq<W, L, SH::CH>(fn, B, tau);
        }
        if constexpr (SH::BLOCKS) {
            bfwd_all<W, L, L, 0, true>(v, 0u, tau, S, gid, stw, a.c);
            block_products<W, R>(v, G::base(last, tau), stw, a.c);
            if constexpr (STAGE) {
                group_sync<T>(gid);
                if (more) stage_seq<W, L, SH::CH>(gn, S + BG::ROWP, tau);
            }
            bdit_all<W, L, last>(v[0], tau, S, gid, stw, a.c);
            if constexpr (STAGE) {
                cp_async_wait();
                group_sync<T>(gid);
            }
            if constexpr (WHOLE) {
                constexpr int VEC = row_vec<W, R>();
                const bool wide = ((uintptr_t)hp & 15u) == 0;
#pragma unroll
                for (int k = 0; k < R; k += VEC) {          // VEC positions of one block: consecutive outputs
                    W t[VEC];
#pragma unroll
                    for (int e = 0; e < VEC; ++e) t[e] = canon<W>(v[0][k + e], a.c.cB, a.c.cBp, a.c.m);
                    st_vec<W, VEC>(hp + block_out<L>((uint32_t)k), t, wide);
                }
                continue;
            }
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const uint32_t x = b0 + ((uint32_t)k << lo0);
                st_out<X>(hp, a.pair0 + rho, N, block_out<L>(x), canon<W>(v[0][k], a.c.cB, a.c.cBp, a.c.m), xa, a.c);
            }
        } else {                                            // one thread per pair, no exchange
            fwd_all<W, L, L, 0, 2, TW_SMEM, true>(v, 0u, tau, S, gid, stw, a.c);
#pragma unroll
            for (int k = 0; k < R; ++k) v[0][k] = pointwise(v[0][k], v[1][k], a.c);
            dit_levels<W, L, 0, TW_SMEM>(v[0], stw, a.c);
#pragma unroll
            for (int k = 0; k < R; ++k)
                st_out<X>(hp, a.pair0 + rho, N, (N - (uint32_t)k) & (N - 1u), canon<W>(v[0][k], (W)1, a.c.onep, a.c.m), xa, a.c);
        }
    }
}

template <typename W, int L, int SRC, int BLK = BLOCK>
__global__ void __launch_bounds__(BLK, BLOCK / BLK) k_conv_fused(const __grid_constant__ RowArgs<W> a)
{
    constexpr int GPC = FusedShape<W, L, BLK>::GPC;
    conv_fused_body<W, L, SRC, NoExact, BLK>(a, (long long)blockIdx.x * GPC, (long long)gridDim.x * GPC);
}

// ---- column/row fused kernel ---------------------------------------------
//
// For 2^RW < N <= 2^LR_max (RW = log2 of the 32 x R elements one warp holds:
// 10 for 32-bit words), the index splits into LC = L - RW top bits and RW low
// bits.  The forward tree's first LC levels act on "columns" (fixed low bits,
// 2^LC elements each): each thread holds whole columns in registers, whose
// node twiddles are the first 2^LC - 1 table entries for every column.  One
// block-wide transpose through shared memory then gives every warp a
// contiguous "row" of 2^RW elements, whose remaining levels (and the first
// RW levels of the inverse) need only warp-level exchanges, so warps run
// independently and one warp's exchanges overlap another's arithmetic.  The
// inverse's last LC levels act on columns again; their twiddles are the runs
// z_{brv_RW(c) 2^J + t}.  Shared memory holds, per row, the f and g slices
// side by side (stride ROWP of the row geometry).

// Forward node levels of one column of RC = 2^LC elements stored at v[OFF ..].
// The column's top bit sits at global level DG0 (0 when the columns hold the
// top bits of the whole transform); node indices at the level of register
// bit J are nbase_J + (k >> (J + 1)), with nbase_J = rowbase >> (J + 1) for
// a row that is itself part of a longer transform (rowbase = its global
// index offset divided by 2^RW).
template <typename W, int LC, int OFF, int J, int DG0, int TWS, int RR>
__device__ __forceinline__ void colf_levels(W (&v)[RR], uint32_t rowbase, const W *__restrict__ tw, const ModC<W> &c)
{
    if constexpr (J >= 0) {
        constexpr int RC = 1 << LC;
        constexpr int dg = DG0 + LC - 1 - J;
        if constexpr (dg == 0) {
#pragma unroll
            for (int k = 0; k < RC; ++k) {
                if (k & (1 << J)) continue;
                ct_bfly_one<W>(v[OFF + k], v[OFF + (k | (1 << J))], c);
            }
        } else {
            constexpr int CNT = RC >> (J + 1);
            constexpr int CH = (CNT >= 2 && tw_per_chunk<W>() == 2) ? 2 : 1;
            const uint32_t nbase = rowbase >> (J + 1);
#pragma unroll
            for (int t0 = 0; t0 < CNT; t0 += CH) {
                W z[CH], zp[CH];
                load_tw<W, CH, TWS>(tw, nbase, (uint32_t)t0, z, zp);
#pragma unroll
                for (int tt = 0; tt < CH; ++tt)
#pragma unroll
                    for (int j = 0; j < (1 << J); ++j) {
                        const int k = ((t0 + tt) << (J + 1)) | j;
                        // whole sequence: node 0 has the twiddle 1 (bounds: ntt_block.cuh)
                        if (DG0 == 0 && dg <= 2 && t0 + tt == 0) ct_bfly_unit<W>(v[OFF + k], v[OFF + (k | (1 << J))], c.m << dg);
                        else ct_bfly<W>(v[OFF + k], v[OFF + (k | (1 << J))], z[tt], zp[tt], c);
                    }
            }
        }
        colf_levels<W, LC, OFF, J - 1, DG0, TWS, RR>(v, rowbase, tw, c);
    }
}

// Transposed (inverse-direction) node levels of one column, deepest first:
// the exact reverse of colf_levels with the same twiddles.  Inputs < 2m,
// outputs < 2m.
template <typename W, int LC, int OFF, int J, int DG0, int TWS, int RR>
__device__ __forceinline__ void colg_levels(W (&v)[RR], uint32_t rowbase, const W *__restrict__ tw, const ModC<W> &c)
{
    if constexpr (J < LC) {
        constexpr int RC = 1 << LC;
        constexpr int dg = DG0 + LC - 1 - J;
        if constexpr (dg == 0) {
#pragma unroll
            for (int k = 0; k < RC; ++k) {
                if (k & (1 << J)) continue;
                gs_bfly_one<W>(v[OFF + k], v[OFF + (k | (1 << J))], c);
            }
        } else {
            constexpr int CNT = RC >> (J + 1);
            constexpr int CH = (CNT >= 2 && tw_per_chunk<W>() == 2) ? 2 : 1;
            const uint32_t nbase = rowbase >> (J + 1);
#pragma unroll
            for (int t0 = 0; t0 < CNT; t0 += CH) {
                W z[CH], zp[CH];
                load_tw<W, CH, TWS>(tw, nbase, (uint32_t)t0, z, zp);
#pragma unroll
                for (int tt = 0; tt < CH; ++tt)
#pragma unroll
                    for (int j = 0; j < (1 << J); ++j) {
                        const int k = ((t0 + tt) << (J + 1)) | j;
                        gs_bfly<W>(v[OFF + k], v[OFF + (k | (1 << J))], z[tt], zp[tt], c);
                    }
            }
        }
        colg_levels<W, LC, OFF, J + 1, DG0, TWS, RR>(v, rowbase, tw, c);
    }
}

template <typename W, int LC, int JC, int CPT, int DG0, int TWS, int RR>
__device__ __forceinline__ void colg_all(W (&v)[RR], uint32_t rowbase, const W *__restrict__ tw, const ModC<W> &c)
{
    if constexpr (JC < CPT) {
        colg_levels<W, LC, JC * (1 << LC), 0, DG0, TWS, RR>(v, rowbase, tw, c);
        colg_all<W, LC, JC + 1, CPT, DG0, TWS, RR>(v, rowbase, tw, c);
    }
}

// All columns JC .. CPT-1 held by a thread (column j at v[j * 2^LC ..]).
template <typename W, int LC, int JC, int CPT, int DG0, int TWS, int RR>
__device__ __forceinline__ void colf_all(W (&v)[RR], uint32_t rowbase, const W *__restrict__ tw, const ModC<W> &c)
{
    if constexpr (JC < CPT) {
        colf_levels<W, LC, JC * (1 << LC), LC - 1, DG0, TWS, RR>(v, rowbase, tw, c);
        colf_all<W, LC, JC + 1, CPT, DG0, TWS, RR>(v, rowbase, tw, c);
    }
}

template <typename W, int LC, int RW, int VEC, int TPP, int JC, int NV, int RR>
__device__ __forceinline__ void bcold_all(W (&v)[RR], uint32_t ptau, const W *__restrict__ tw, const ModC<W> &c)
{
    if constexpr (JC < NV) {
        const uint32_t col = VEC * (ptau + (uint32_t)JC * TPP);
        bcold_levels<W, LC, VEC, JC * VEC * (1 << LC), 0, RR>(v, __brev(col >> BB) >> (32 - (RW - BB)), tw, c);
        bcold_all<W, LC, RW, VEC, TPP, JC + 1, NV, RR>(v, ptau, tw, c);
    }
}

// A row group of the column/row kernels: TPP threads hold one sequence pair
// of 2^LROW elements, as RC rows of 2^RW.  FULL (whole sequences): block
// form, rows padded for vector access, the first N / 8 pairs of the table in
// shared memory, VEC adjacent columns per thread access.  Otherwise (rows of
// the split path's row-twiddle form): the complete transform, twiddles from
// the plan's table.
template <typename W, int LROW, bool FULL, int BLK = BLOCK>
struct CRShape {
    static constexpr int RW = Arith<W>::RB + 5;
    static constexpr int LC = LROW - RW;                    // column bits inside one row
    static constexpr int RC = 1 << LC;
    static constexpr int ROWP = FULL ? BGeo<W, RW>::ROWP : Geo<W, RW>::ROWP;
    static constexpr int TPP = 32 * RC;                     // threads per row
    static constexpr int PPC = BLK / TPP;                   // rows per block
    static_assert(PPC >= 1, "a row needs more threads than the block has");
    static constexpr int CPT = (1 << RW) / TPP;             // columns per thread
    static constexpr int VEC = CPT < (int)(16 / sizeof(W)) ? CPT : (int)(16 / sizeof(W));
    static constexpr int TWL = LROW - BB;                   // TwBytes: 2^(TWL - 1) pairs
    static constexpr size_t tw_bytes = FULL ? TwBytes<W, TWL>::v : 0;
    static constexpr size_t rows_bytes = (size_t)PPC * RC * 2 * ROWP * sizeof(W);
    static constexpr bool STAGE = FULL && sizeof(W) == 4;   // the next pair staged by asynchronous copies
    static constexpr size_t smem = tw_bytes + rows_bytes + (STAGE ? (size_t)PPC * (sizeof(W) << LROW) : 0);   // and its g
};

// One row of 2^RW words by a warp's asynchronous copies, to a padded or a
// plain row in shared memory; 16 bytes each where source and layout allow.
template <typename W, int RW, bool PADDED>
__device__ __forceinline__ void stage_row(const W *src, W *dst, uint32_t lane)
{
    using GR = BGeo<W, RW>;
    constexpr uint32_t Q = (uint32_t)(16 / sizeof(W));
    if ((GR::VX || !PADDED) && ((uintptr_t)src & 15u) == 0) {
#pragma unroll
        for (uint32_t i = 0; i < (1u << RW) / (32 * Q); ++i) {
            const uint32_t e = (lane + 32u * i) * Q;
            cp_async<16>(dst + (PADDED ? GR::pad(e) : e), src + e);
        }
    } else {
#pragma unroll 8
        for (uint32_t i = 0; i < (1u << RW) / 32; ++i) {
            const uint32_t e = lane + 32u * i;
            cp_async<sizeof(W)>(dst + (PADDED ? GR::pad(e) : e), src + e);
        }
    }
}

// A thread's columns (VEC adjacent ones at VEC ptau + j VEC TPP, 2^LC
// elements each) from rows in shared memory.
template <typename W, int RW, int LC, int VEC, int TPP, bool PADDED, int R>
__device__ __forceinline__ void cols_from_rows(const W *S, uint32_t stride, uint32_t ptau, W (&v)[R])
{
    using GR = BGeo<W, RW>;
#pragma unroll
    for (int j = 0; j < (R >> LC) / VEC; ++j)
#pragma unroll
        for (int k = 0; k < (1 << LC); ++k) {
            const uint32_t c = VEC * (ptau + (uint32_t)j * TPP);
            W t[VEC];
            ld_vec<W, VEC>(S + (size_t)k * stride + (PADDED ? GR::pad(c) : c), t, GR::VX || !PADDED);
#pragma unroll
            for (int e = 0; e < VEC; ++e) v[((j * VEC + e) << LC) + k] = t[e];
        }
}

// Column/row fused convolution of whole sequences (f, g, h or the descriptor
// list), by blocks (ntt_block.cuh).
// Rows [base + row group, end) by steps of stride; end is a.nrows unless ITEM.
// OUT 0: canonical, at block_out(x) (a whole convolution); OUT 1: lazy
// residues of a row of a convolution's split path, after the twist, stored
// in place: position 4 t' + r holds the inverse's element <4 t' - r> of the
// row (row_element below; the transposed column pass accounts for it); the
// factor 2^(B + BB) / N is in the twist's diagonal.
template <typename W, int L, int SRC, bool ITEM = false, int OUT = 0, class X = NoExact, int BLK = BLOCK>
__device__ __forceinline__ void conv_cr_body(const RowArgs<W> &a, long long base, long long stride, long long end = 0,
                                             const ExactFused *xa = nullptr)
{
    using SH = CRShape<W, L, true, BLK>;
    constexpr int RW = SH::RW, LC = SH::LC, RC = SH::RC, TPP = SH::TPP, PPC = SH::PPC, CPT = SH::CPT, VEC = SH::VEC;
    using GR = BGeo<W, RW>;
    constexpr int R = GR::R;
    static_assert(LC >= 1 && CPT * RC == R, "column/row split");
    constexpr uint32_t N = 1u << L;
    constexpr int last = GR::NPASS - 1;
    constexpr bool STAGE = SH::STAGE && !X::IN64 && SRC != 2;
    constexpr uint32_t INB = X::IN64 ? 8u : (uint32_t)sizeof(W);     // bytes per input element
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int pid = threadIdx.x / TPP;
    const uint32_t ptau = threadIdx.x % TPP;
    const int wr = (int)(ptau >> 5);
    const uint32_t lane = ptau & 31u;
    W *stw = reinterpret_cast<W *>(smem_raw);
    W *P = reinterpret_cast<W *>(smem_raw + SH::tw_bytes) + (size_t)pid * RC * 2 * GR::ROWP;
    W *Srow = P + (size_t)wr * 2 * GR::ROWP;                // this warp's g slice (also H); f slice follows
    stage_twiddles<W>(a.tw, stw, TwBytes<W, SH::TWL>::pairs);
    __syncthreads();

    // The row groups of a block synchronise block-wide and step through the
    // rows in rounds together (a group whose row of the round is past the
    // end skips its memory accesses), so every group runs the same phase at
    // the same time: measured 9% (2^11) and 15% (2^12) faster than a
    // barrier per group, whose groups drift apart across the unrolled code.
    auto psync = [&]() { __syncthreads(); };
    auto ptrs = [&](long long rho, const W *&fp, const W *&gp, W *&hp) {
        const long long pair = a.pair0 + rho;
        if constexpr (SRC == 1) {
            const DevDesc<W> d = a.descs[pair];
            fp = d.f; gp = d.g; hp = d.h;
        } else {
            fp = seq_base<X>(a.f, pair, N); gp = seq_base<X>(a.g, pair, N);
            hp = X::GARNER ? nullptr : a.h + (size_t)pair * N;
        }
    };
    // A thread's columns: VEC adjacent ones at VEC ptau + j VEC TPP; column c
    // holds the elements c + k 2^RW, k < RC, in registers (j VEC + e) RC + k.
    auto col_of = [&](int j) { return VEC * (ptau + (uint32_t)j * TPP); };
    auto load_cols = [&](const W *src, W (&dst)[R]) {       // from global memory (X::IN64: reduced on the way)
        auto all = [&](bool wide) {
#pragma unroll
            for (int j = 0; j < CPT / VEC; ++j)
#pragma unroll
                for (int k = 0; k < RC; ++k) {
                    const uint32_t x = col_of(j) + ((uint32_t)k << RW);
                    W t[VEC];
                    if constexpr (X::IN64) {
                        ld_residues<VEC>(reinterpret_cast<const long long *>(src) + x, t, wide, xa, a.c);
                    } else {
                        ld_vec<W, VEC>(src + x, t, wide);
                    }
#pragma unroll
                    for (int e = 0; e < VEC; ++e) dst[(j * VEC + e) * RC + k] = t[e];
                }
        };
        if (VEC > 1 && ((uintptr_t)src & (X::IN64 ? 15u : VEC * sizeof(W) - 1)) == 0) all(true);
        else all(false);
    };
    auto store_cols = [&](const W (&v)[R], W *S) {          // into the rows' slices
#pragma unroll
        for (int j = 0; j < CPT / VEC; ++j)
#pragma unroll
            for (int k = 0; k < RC; ++k) {
                W t[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) t[e] = v[(j * VEC + e) * RC + k];
                st_vec<W, VEC>(S + (size_t)k * 2 * GR::ROWP + GR::pad(col_of(j)), t, GR::VX);
            }
    };
    // STAGE (32-bit words): the next pair arrives by asynchronous copies
    // while this one is convolved: each warp brings its own row of f into its
    // f slice (free after the block products) and of g into the staging rows
    // G (read before the first barrier); the wait before the second barrier
    // makes both visible to the columns of the next round.  No register
    // holds loaded words across the inverse, and no load waits on L2:
    // measured on GB300, 4096 x 2^14 412 -> 394 us at equal clocks (without
    // any global load: 369), 8192 x 2^13 392 -> 376, 2^12 1.5%, 2^11 equal.
    // 64-bit words, whose padded rows take 8-byte copies only, lose by it
    // (301 x 2^13: 59.4 -> 61.5 us), and so do inputs in host memory (SRC 2),
    // whose copies all SMs would issue and wait for at the same time (256 x
    // 2^14 over C2C 254 -> 301 us); there the next f is loaded into registers
    // after the block products, and g while f's columns are transformed.
    W *G = reinterpret_cast<W *>(smem_raw + SH::tw_bytes + SH::rows_bytes) + ((size_t)pid << L);
    auto stage_f = [&](const W *f) { stage_row<W, RW, true>(f + ((size_t)wr << RW), Srow + GR::ROWP, lane); };
    auto stage_g = [&](const W *g) { stage_row<W, RW, false>(g + ((size_t)wr << RW), G + ((size_t)wr << RW), lane); };
    const long long lim = ITEM ? end : a.nrows;
    W v[2][R];
    const W *fp = nullptr, *gp = nullptr;
    W *hp = nullptr;
    if (base + pid < lim) {
        ptrs(base + pid, fp, gp, hp);
        if constexpr (STAGE) {
            stage_f(fp);
            stage_g(gp);
        } else {
            load_cols(fp, v[1]);
        }
    }
    if constexpr (STAGE) {
        cp_async_wait();
        psync();
    }
    for (long long round = base; round < lim; round += stride) {
        const long long rho = round + pid;
        const bool live = PPC == 1 || rho < lim;            // this group's row of the round exists
        const bool more = rho + stride < lim;
        W *const hcur = hp;
        if constexpr (!STAGE) {
            if (ptau == 0 && more) {
                const W *fn, *gn;
                W *hn;
                ptrs(rho + stride, fn, gn, hn);
                prefetch_l2(fn, N * INB);
                prefetch_l2(gn, N * INB);
            }
            if (live) load_cols(gp, v[0]);
        }
        // forward, column phase.
        // No barrier before the column stores: in the slices every thread
        // writes only the positions of its own columns, which it alone read
        // here (f) or in the previous row's inverse column phase (g).
        if constexpr (STAGE) cols_from_rows<W, RW, LC, VEC, TPP, true>(P + GR::ROWP, 2 * GR::ROWP, ptau, v[1]);
        colf_all<W, LC, 0, CPT, 0, TW_SMEM, R>(v[1], 0u, stw, a.c);
        store_cols(v[1], P + GR::ROWP);
        if constexpr (STAGE) cols_from_rows<W, RW, LC, VEC, TPP, false>(G, 1u << RW, ptau, v[0]);
        colf_all<W, LC, 0, CPT, 0, TW_SMEM, R>(v[0], 0u, stw, a.c);
        store_cols(v[0], P);
        psync();
        if (more) {
            ptrs(rho + stride, fp, gp, hp);
            if constexpr (STAGE) stage_g(gp);
        }
        // row phase (warp wr owns row wr of this row group): forward, block
        // products, inverse
        bload<W, RW, 0>(v[0], Srow, lane);
        bload<W, RW, 0>(v[1], Srow + GR::ROWP, lane);
        bfwd_all<W, L, RW, 0, false>(v, (uint32_t)wr << RW, lane, Srow, 0, stw, a.c);
        block_products<W, R>(v, ((uint32_t)wr << RW) + GR::base(last, lane), stw, a.c);
        if (more) {
            if constexpr (STAGE) {
                __syncwarp();
                stage_f(fp);
            } else {
                load_cols(fp, v[1]);
            }
        }
        bdit_all<W, RW, last>(v[0], lane, Srow, 0, stw, a.c);
        bstore<W, RW, 0>(v[0], Srow, lane);
        if constexpr (STAGE) cp_async_wait();
        psync();
        // inverse, column phase
        W r0[X::GARNER == 2 ? R : 1];                       // the first prime's residues of this thread's outputs
        if constexpr (X::GARNER == 2) {
            const uint32_t *prev = xa->prev + (size_t)(a.pair0 + (live ? rho : base)) * N;
#pragma unroll
            for (int j = 0; j < CPT / VEC; ++j)
#pragma unroll
                for (int k = 0; k < RC; ++k) {
                    uint32_t t[VEC];                        // (the plan's scratch: aligned)
                    ld_vec<uint32_t, VEC>(prev + block_out<L>(col_of(j) + ((uint32_t)k << RW)), t, true);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) r0[(j * RC + k) * VEC + e] = t[e];
                }
        }
        cols_from_rows<W, RW, LC, VEC, TPP, true>(P, 2 * GR::ROWP, ptau, v[0]);
        bcold_all<W, LC, RW, VEC, TPP, 0, CPT / VEC, R>(v[0], ptau, stw, a.c);
        if (!live) continue;                                // (no barrier follows in this round)
        const bool wide = X::GARNER > 0 ? ((uintptr_t)xa->h64 & 15u) == 0 : ((uintptr_t)hcur & (VEC * sizeof(W) - 1)) == 0;
#pragma unroll
        for (int j = 0; j < CPT / VEC; ++j)
#pragma unroll
            for (int k = 0; k < RC; ++k) {
                const uint32_t x = col_of(j) + ((uint32_t)k << RW);
                W t[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) t[e] = v[0][(j * VEC + e) * RC + k];
                if constexpr (OUT == 1) {
                    st_vec<W, VEC>(hcur + x, t, true);      // scratch rows: aligned
                } else {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) t[e] = canon<W>(t[e], a.c.cB, a.c.cBp, a.c.m);
                    if constexpr (X::GARNER > 0) {
                        st_garner<X::GARNER, VEC>((size_t)(a.pair0 + rho) * N + block_out<L>(x), t, r0 + (X::GARNER == 2 ? (j * RC + k) * VEC : 0), wide, xa, a.c);
                    } else {
                        st_vec<W, VEC>(hcur + block_out<L>(x), t, wide);
                    }
                }
            }
    }
}

template <typename W, int L, int SRC, int OUT = 0, int BLK = BLOCK>
__global__ void __launch_bounds__(BLK, BLOCK / BLK) k_conv_cr(const __grid_constant__ RowArgs<W> a)
{
    constexpr int PPC = CRShape<W, L, true, BLK>::PPC;
    conv_cr_body<W, L, SRC, false, OUT, NoExact, BLK>(a, (long long)blockIdx.x * PPC, (long long)gridDim.x * PPC);
}

// Rows of the split path's row-twiddle form: one row of 2^LROW elements of
// the length-2^L tree per row group, inputs F~, G~ and output H~ (lazy
// residues, natural order) in the wave's scratch.  The node twiddles depend
// on the row and are read from the plan's table; the inverse is the
// transposed tree, whose twiddles (like the forward ones) are contiguous
// runs of it.  The complete transform with a pointwise product.
template <typename W, int L, int LROW>
__global__ void __launch_bounds__(BLOCK, 1) k_conv_rows(const __grid_constant__ RowArgs<W> a)
{
    using SH = CRShape<W, LROW, false>;
    using GR = Geo<W, SH::RW>;
    constexpr int RW = SH::RW, LC = SH::LC, RC = SH::RC, TPP = SH::TPP, PPC = SH::PPC, CPT = SH::CPT;
    constexpr int R = GR::R;
    static_assert(PPC == 1 && LC >= 1 && CPT * RC == R, "one row per block");
    constexpr uint32_t N = 1u << L;
    constexpr int last = GR::NPASS - 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t ptau = threadIdx.x;
    const int wr = (int)(ptau >> 5);
    const uint32_t lane = ptau & 31u;
    W *P = reinterpret_cast<W *>(smem_raw);
    W *Srow = P + (size_t)wr * 2 * GR::ROWP;                // this warp's g slice (also H); f slice follows
    const uint32_t b0 = GR::base(0, lane);
    constexpr int lo0 = GR::lo(0);
    for (long long rho = blockIdx.x; rho < a.nrows; rho += gridDim.x) {
        const uint32_t row = (uint32_t)rho & ((1u << (L - LROW)) - 1u);
        const size_t off = (size_t)(rho >> (L - LROW)) * N + ((size_t)row << LROW);
        const W *fp = a.f + off, *gp = a.g + off;
        W *hp = a.h + off;
        const uint32_t rowoff = row << LROW;
        W v[2][R];
        auto load_cols = [&](const W *src, W (&dst)[R]) {
#pragma unroll
            for (int j = 0; j < CPT; ++j)
#pragma unroll
                for (int k = 0; k < RC; ++k) dst[j * RC + k] = src[ptau + (uint32_t)j * TPP + ((uint32_t)k << RW)];
        };
        auto store_cols = [&](const W (&s)[R], W *S) {
#pragma unroll
            for (int j = 0; j < CPT; ++j)
#pragma unroll
                for (int k = 0; k < RC; ++k) S[(size_t)k * 2 * GR::ROWP + GR::pad(ptau + (uint32_t)j * TPP)] = s[j * RC + k];
        };
        load_cols(fp, v[1]);
        if (ptau == 0 && rho + gridDim.x < a.nrows) {
            const long long nx = rho + gridDim.x;
            const size_t no = (size_t)(nx >> (L - LROW)) * N + ((size_t)((uint32_t)nx & ((1u << (L - LROW)) - 1u)) << LROW);
            prefetch_l2(a.f + no, (uint32_t)(sizeof(W) << LROW));
            prefetch_l2(a.g + no, (uint32_t)(sizeof(W) << LROW));
        }
        load_cols(gp, v[0]);
        // (no barrier before the column stores: see conv_cr_body)
        colf_all<W, LC, 0, CPT, L - LROW, TW_GLOBAL, R>(v[1], rowoff >> RW, a.tw, a.c);
        store_cols(v[1], P + GR::ROWP);
        colf_all<W, LC, 0, CPT, L - LROW, TW_GLOBAL, R>(v[0], rowoff >> RW, a.tw, a.c);
        store_cols(v[0], P);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const uint32_t y = b0 + ((uint32_t)k << lo0);
            v[0][k] = Srow[GR::pad(y)];
            v[1][k] = Srow[GR::ROWP + GR::pad(y)];
        }
        fwd_all<W, L, RW, 0, 2, TW_GLOBAL>(v, rowoff + ((uint32_t)wr << RW), lane, Srow, 0, a.tw, a.c);
#pragma unroll
        for (int k = 0; k < R; ++k) v[0][k] = pointwise(v[1][k], v[0][k], a.c);
        inv_all<W, L, RW, last, TW_GLOBAL>(v[0], rowoff + ((uint32_t)wr << RW), lane, Srow, 0, a.tw, a.c);
#pragma unroll
        for (int k = 0; k < R; ++k) Srow[GR::pad(b0 + ((uint32_t)k << lo0))] = v[0][k];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const uint32_t col = ptau + (uint32_t)j * TPP;
#pragma unroll
            for (int k = 0; k < RC; ++k) v[0][j * RC + k] = P[(size_t)k * 2 * GR::ROWP + GR::pad(col)];
        }
        colg_all<W, LC, 0, CPT, L - LROW, TW_GLOBAL, R>(v[0], rowoff >> RW, a.tw, a.c);
#pragma unroll
        for (int j = 0; j < CPT; ++j)
#pragma unroll
            for (int k = 0; k < RC; ++k) hp[ptau + (uint32_t)j * TPP + ((uint32_t)k << RW)] = v[0][j * RC + k];
    }
}

// The exact convolution's fused launches (whole sequences, contiguous; h goes
// to e.h64 as signed integers).  X = ExactOne: the whole convolution of a
// plan of one prime, 24 bytes per element instead of 48.  X = ExactLast: the
// second of two primes from its residues, reconstructing from its own and
// the first one's result, 60 bytes instead of 72; reading the inputs in both
// primes' kernels (48 bytes) measured 321 us against 303 at 4096 x 2^12
// (separate passes 318), since 64-bit inputs leave no shared memory to stage
// them in.
template <typename W, int L, class X, int BLK>
__global__ void __launch_bounds__(BLK, BLOCK / BLK) k_conv_exact(const __grid_constant__ RowArgs<W> a,
                                                                const __grid_constant__ ExactFused e)
{
    constexpr int RW = Arith<W>::RB + 5;
    if constexpr (L <= RW) {
        constexpr int GPC = FusedShape<W, L, BLK>::GPC;
        conv_fused_body<W, L, 0, X, BLK>(a, (long long)blockIdx.x * GPC, (long long)gridDim.x * GPC, &e);
    } else {
        constexpr int PPC = CRShape<W, L, true, BLK>::PPC;
        conv_cr_body<W, L, 0, false, 0, X, BLK>(a, (long long)blockIdx.x * PPC, (long long)gridDim.x * PPC, 0, &e);
    }
}

// ---- one persistent launch for every whole-sequence length of a batch ----
//
// Work items {log2 N, first pair, count} of a batch plan's descriptor list
// (grouped by length) are pulled by the blocks with an atomic counter; a
// block runs the item with the fused body of its length, staging that
// length's twiddle table into shared memory first.  Blocks never wait on
// one another.

struct WorkItem {
    int L;
    int reserved;
    long long first;
    long long count;
};

// The per-length arguments (descriptor list, twiddle table, constants) travel
// by value in the kernel's parameter space, so each length's body reads them
// as constant-bank operands, as the single-length kernels do, instead of
// holding them in registers.
template <typename W> struct PersistArgs {
    const WorkItem *items;
    int nitems;
    int *counter;                      // zeroed before each launch
    RowArgs<W> cls[LRMax<W>::v + 1];   // indexed by log2 N
};

template <typename W, int L>
__device__ __forceinline__ void persist_item(const PersistArgs<W> &a, const WorkItem &w)
{
    constexpr int RW = Arith<W>::RB + 5;
    // rows [first, first + count) of the descriptor list; the one-warp body
    // takes them as a local copy of its arguments with nrows set, the
    // column/row body as an explicit bound.  (64-bit words of up to 2^9: 144
    // bytes of spills where the complete transform had 24, and faster all the
    // same, on GB300: 61440 pairs of 2^6 .. 2^9 177 -> 166 us, 8192 x 2^9 111
    // -> 104, 16384 x 2^8 95 -> 90, 1200 pairs 45.6 -> 43.2.)
    if constexpr (L <= RW) {
        RowArgs<W> ra = a.cls[L];
        ra.nrows = w.first + w.count;
        conv_fused_body<W, L, 1>(ra, w.first, FusedShape<W, L>::GPC);
    }
    else conv_cr_body<W, L, 1, true>(a.cls[L], w.first, CRShape<W, L, true>::PPC, w.first + w.count);
}

template <typename W, int L, int HI>
__device__ __forceinline__ void persist_dispatch(const PersistArgs<W> &a, const WorkItem &w)
{
    if constexpr (L <= HI) {
        if (w.L == L) persist_item<W, L>(a, w);
        else persist_dispatch<W, L + 1, HI>(a, w);
    }
}

// HI: the longest length the kernel is compiled for (the one-warp lengths
// only, or every whole-sequence length).
template <typename W, int HI>
__global__ void __launch_bounds__(BLOCK, 1) k_conv_persistent(const __grid_constant__ PersistArgs<W> a)
{
    __shared__ int item;
    for (;;) {
        __syncthreads();                                   // previous item done with shared memory
        if (threadIdx.x == 0) item = atomicAdd(a.counter, 1);
        __syncthreads();
        const int it = item;
        if (it >= a.nitems) break;
        persist_dispatch<W, 0, HI>(a, a.items[it]);
    }
}

// Natural-order forward transform (Eq. 2) or inverse transform (Eq. 3) of
// whole sequences (L <= LR_max).  The forward tree leaves X(brv(x)) at x; a
// shared-memory pass puts it back in natural order.  The inverse is
// N^-1 R F: same forward tree, output index <-u>_N, factor N^-1.
template <typename W> struct NttArgs {
    const W *x;
    W *y;
    long long batch;
    const W *tw;
    ModC<W> c;
};

// Rows of the natural-order kernels: one row per group of T threads for the
// exchanges, and a plain one that holds the group's next sequence, brought
// by asynchronous copies while this one is transformed.  Measured on GB300
// against loading it into registers: 4096 x 2^14 forward 177 -> 169 us, 2^13
// 155 -> 147; 64-bit words 2048 x 2^13, which had no registers to spare for
// it, 160 -> 150.  (Two groups of 512 threads with 64 registers each instead
// of one: 226 us at 2^14; two alternating exchange rows, which need half the
// barriers: 190 -- the warps drift apart across the unrolled code.)
template <typename W, int L> struct NttShape {
    using G = Geo<W, L>;
    static constexpr int GPC = BLOCK / G::T;
    // Staged sequences of rows that share a warp lie NB words apart: T (or a
    // 16-byte copy's words) more than their length, so that the rows' runs of
    // T words fall on different banks: 149797 x 2^6 44.0 -> 32.9 us, 74899 x
    // 2^7 26.9 -> 21.5, 37450 x 2^8 19.5 -> 17.5; 64-bit words 299594 x 2^5
    // 52.1 -> 42.6, 149797 x 2^6 39.6 -> 36.0.
    static constexpr int Q = (int)(16 / sizeof(W));
    static constexpr int NB = G::ROW + (G::T >= (int)(128 / sizeof(W)) ? 0 : G::T > Q ? G::T : Q);
    static constexpr size_t rows = TwBytes<W, L>::v, next = rows + ((size_t)GPC * G::ROWP * sizeof(W) + 15) / 16 * 16;
    static constexpr size_t smem = G::T == 1 ? rows : next + (size_t)GPC * NB * sizeof(W);
};

// One transform of the loop these kernels share: the staged sequence through
// the forward tree, the next one's copies issued once every thread of the
// group has read this one; v in the last pass's layout.  (The group's first
// sequence straight into registers, for batches of one sequence per group:
// 4096 x 2^14 169 -> 176 us, not kept.)
template <typename W, int L, class Next>
__device__ __forceinline__ void staged_forward(W (&v)[1][Geo<W, L>::R], const W *B, W *S, uint32_t tau, int gid, const W *stw,
                                               const ModC<W> &c, Next next)
{
    using G = Geo<W, L>;
    const uint32_t b0 = G::base(0, tau);
#pragma unroll
    for (int k = 0; k < G::R; ++k) v[0][k] = B[b0 + ((uint32_t)k << G::lo(0))];
    fwd_pass<W, L, L, 0, 1, TW_SMEM, true>(v, b0, stw, c);
    exchange<W, L, 0, 1, 1>(v, S, tau, gid);
    next();
    fwd_all<W, L, L, 1, 1, TW_SMEM, true>(v, 0u, tau, S, gid, stw, c);
}

template <typename W, int L, bool INV>
__global__ void __launch_bounds__(BLOCK, 1) k_ntt_rows(const __grid_constant__ NttArgs<W> a)
{
    using G = Geo<W, L>;
    using SH = NttShape<W, L>;
    constexpr int T = G::T, R = G::R, GPC = SH::GPC;
    constexpr uint32_t N = 1u << L, Q = (uint32_t)(16 / sizeof(W));
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gid = threadIdx.x / T;
    const uint32_t tau = threadIdx.x % T;
    W *stw = reinterpret_cast<W *>(smem_raw);
    W *S = reinterpret_cast<W *>(smem_raw + SH::rows) + (size_t)gid * G::ROWP;
    W *B = reinterpret_cast<W *>(smem_raw + SH::next) + (size_t)gid * SH::NB;
    const uint32_t b0 = G::base(0, tau);
    stage_twiddles<W>(a.tw, stw, TwBytes<W, L>::pairs);
    const long long step = (long long)gridDim.x * GPC;
    long long rho = (long long)blockIdx.x * GPC + gid;
    if constexpr (T == 1) {
        // One thread per sequence: read and written by 16 bytes, reordered
        // in registers, the next one loaded ahead.  Measured on GB300 against
        // staging and reordering in shared memory, whose rows of N words
        // share banks: 1198373 x 2^3 30.2 -> 12.5 us, 299594 x 2^5 62 -> 20.6;
        // 64-bit words 1198373 x 2^3 58.7 -> 28.4, 599187 x 2^4 69.4 -> 41.2.
        constexpr int VEC = row_vec<W, R>();
        W w[R];
        if (rho < a.batch) ld_row<W, R>(a.x + (size_t)rho * N, w);
        __syncthreads();
        for (; rho < a.batch; rho += step) {
            W v[1][R];
#pragma unroll
            for (int k = 0; k < R; ++k) v[0][k] = w[k];
            if (rho + step < a.batch) ld_row<W, R>(a.x + (size_t)(rho + step) * N, w);
            fwd_pass<W, L, L, 0, 1, TW_SMEM, true>(v, 0u, stw, a.c);
            W *yp = a.y + (size_t)rho * N;
            const bool wide = ((uintptr_t)yp & (VEC * sizeof(W) - 1)) == 0;
#pragma unroll
            for (int t0 = 0; t0 < R; t0 += VEC) {
                W o[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const W x = v[0][brv_c<L>(INV ? (R - t0 - e) & (R - 1) : t0 + e)];
                    o[e] = csub<W>(INV ? shoup_full<W>(x, a.c.ninv, a.c.ninvp, a.c.m) : shoup_one<W>(x, a.c.onep, a.c.m), a.c.m);
                }
                st_vec<W, VEC>(yp + t0, o, wide);
            }
        }
    } else {
        auto stage = [&](long long r) { if (r < a.batch) stage_seq<W, L, Q>(a.x + (size_t)r * N, B, tau); };
        stage(rho);
        cp_async_wait();
        __syncthreads();
        W v[1][R];
        for (; rho < a.batch; rho += step) {
            staged_forward<W, L>(v, B, S, tau, gid, stw, a.c, [&] { stage(rho + step); });
            cp_async_wait();                                // visible after the next two barriers
            group_sync<T>(gid);
            scatter_reversed<W, L>(v[0], S, tau);
            group_sync<T>(gid);
            // output index t = b0 + k T (a warp's stores are one aligned run);
            // the inverse takes its value from <-t>_N
            gather_natural<W, L, INV>(v[0], S, tau);
            W *yp = a.y + (size_t)rho * N;
#pragma unroll
            for (int k = 0; k < R; ++k)
                yp[b0 + ((uint32_t)k << G::lo(0))] = csub<W>(INV ? shoup_full<W>(v[0][k], a.c.ninv, a.c.ninvp, a.c.m)
                                                                 : shoup_one<W>(v[0][k], a.c.onep, a.c.m), a.c.m);
        }
    }
}

// Split path for L > LR: "column" transforms of the top LC = L - LR index
// bits.  Element (c, k) of a sequence is x = c + k 2^LR (c < 2^LR, k < 2^LC);
// every level of the top bits has node index k >> (bits below), the same for
// all columns.  NS sequences per thread (f and g).
template <typename W> struct ColArgs {
    const W *src0;      // SRC == 0: contiguous batch base of sequence 0 (f)
    const W *src1;      // ... of sequence 1 (g)
    const DevDesc<W> *descs;   // SRC == 1
    W *dst0;            // scratch of the wave (F~), [pairs][N]
    W *dst1;            // scratch (G~)
    W *out;             // cols_inv, DST == 0: contiguous output base
    long long npairs;   // pairs in this wave
    long long pair0;    // first pair of the wave in the batch / descriptor list
    const W *tw;
    ModC<W> c;
    const W *pw;        // convolutions: (w^e, Shoup quotient) pairs, e < N (the twist)
    const W *pwl;       // (w^(s l), quotient) at s 32 + l, s < 2^(L-LR), l < 32
    const W *pd;        // one column pass: (w^(brv(k) t), quotient) at x = t + k 2^LR
};

// The row element that position p of a row of 2^LR holds after the rows of
// the twist form (OUT 1 of the column/row kernel).
template <int LR>
__device__ __forceinline__ uint32_t row_element(uint32_t p)
{
    return (p - 2 * (p & ((1u << BB) - 1u))) & ((1u << LR) - 1u);
}

// The four-step twist, one of the two forms of the split path of
// convolutions and natural-order transforms (the plan picks one per word
// size and length; the autotuner measures both).  In the other form the rows
// read their node twiddles, which then depend on the row, from the plan's
// table.  With the twist: after the column levels, element (r, t) -- r the
// top L - LR index bits at their tree position, t the low LR bits -- is
// multiplied by w^(brv(r) t).  That turns every row's remaining levels into
// the length-2^LR transform with the uniform table z'_i = w'^brv(i),
// w' = w^(2^(L-LR)), whose entries are the first 2^(LR-1) of the plan's
// table; the rows then run the whole-sequence convolution kernel (or, for
// transforms, k_rows_uni).  The inverse (the transposed tree) applies the
// same diagonal between the rows and the transposed column levels.  Output
// in [0, 2m).
//
// With one column pass the factor of element x = t + k 2^LR depends on x
// alone (not on the pair), so the plan stores it at x (ColArgs::pd): one
// coalesced, L2-resident vector load and one Shoup product per element.
// With two column passes (k_cols_mid_*) it is split as w^(s t0) w^(s l),
// t = t0 + l, l = t mod 32 (the lane): the first is the same for a warp (one
// broadcast load), the second comes from a small lane table (s, l) ->
// w^(s l), coalesced; two Shoup products.  Each (power, Shoup quotient)
// pair is one vector load.
template <typename W> struct PairVec;
template <> struct PairVec<uint32_t> { using T = uint2; };
template <> struct PairVec<uint64_t> { using T = ulonglong2; };

template <typename W>
__device__ __forceinline__ void ld_pair_g(const W *p, W &z, W &zp)
{
    const typename PairVec<W>::T q = __ldg(reinterpret_cast<const typename PairVec<W>::T *>(p));
    z = q.x; zp = q.y;
}

template <typename W>
__device__ __forceinline__ void ld_pair(const W *p, W &z, W &zp)
{
    const typename PairVec<W>::T q = *reinterpret_cast<const typename PairVec<W>::T *>(p);
    z = q.x; zp = q.y;
}

// The twist factor of (s, t): e = s (t - l) mod N for the warp-uniform part;
// lt is the lane table (shared memory, or the plan's copy).
template <typename W, int L>
__device__ __forceinline__ void twist_factors(uint32_t s, uint32_t t, const ColArgs<W> &a, const W *lt, W &z0, W &z0p,
                                              W &z1, W &z1p)
{
    const uint32_t l = t & 31u;
    const uint32_t e = (s * (t - l)) & ((1u << L) - 1u);
    ld_pair_g<W>(a.pw + 2 * (size_t)e, z0, z0p);
    ld_pair<W>(lt + 2 * ((size_t)s * 32 + l), z1, z1p);
}

template <typename W, int L>
__device__ __forceinline__ W twist(W v, uint32_t s, uint32_t t, const ColArgs<W> &a, const W *lt)
{
    W z0, z0p, z1, z1p;
    twist_factors<W, L>(s, t, a, lt, z0, z0p, z1, z1p);
    return shoup<W>(shoup<W>(v, z1, z1p, a.c.m), z0, z0p, a.c.m);
}

template <int BITS>
__host__ __device__ constexpr uint32_t brv_c32(uint32_t k)
{
    uint32_t r = 0;
    for (int i = 0; i < BITS; ++i) r |= ((k >> i) & 1u) << (BITS - 1 - i);
    return r;
}

// Pairs 0 .. CNT-1 of the plan's table (the same for every column).
template <typename W, int CNT>
__device__ __forceinline__ void load_tw_run(const W *__restrict__ tw, W (&z)[CNT], W (&zp)[CNT])
{
#pragma unroll
    for (int t = 0; t < CNT; ++t) {
        W a[1], ap[1];
        load_tw<W, 1, TW_GLOBAL>(tw, 0u, (uint32_t)t, a, ap);
        z[t] = a[0]; zp[t] = ap[0];
    }
}

template <typename W, int L, int LR, int J>
__device__ __forceinline__ void col_fwd_level(W (&v)[1 << (L - LR)], const W *__restrict__ tw, const ModC<W> &c)
{
    // J = register bit, element bit b = LR + J, global level L - 1 - b
    constexpr int RC = 1 << (L - LR);
    constexpr int dg = L - LR - 1 - J;
    if constexpr (dg == 0) {
#pragma unroll
        for (int k = 0; k < RC; ++k) {
            if (k & (1 << J)) continue;
            ct_bfly_one<W>(v[k], v[k | (1 << J)], c);
        }
    } else {
        constexpr int CNT = RC >> (J + 1);
        W z[CNT], zp[CNT];
        load_tw_run<W, CNT>(tw, z, zp);
#pragma unroll
        for (int k = 0; k < RC; ++k) {
            if (k & (1 << J)) continue;
            ct_bfly<W>(v[k], v[k | (1 << J)], z[k >> (J + 1)], zp[k >> (J + 1)], c);
        }
    }
}

template <typename W, int L, int LR, int J>
__device__ __forceinline__ void col_fwd_levels(W (&v)[1 << (L - LR)], const W *__restrict__ tw, const ModC<W> &c)
{
    if constexpr (J >= 0) {
        col_fwd_level<W, L, LR, J>(v, tw, c);
        col_fwd_levels<W, L, LR, J - 1>(v, tw, c);
    }
}

// Column kernels run blocks of COLB threads and are bound by memory latency:
// what counts is how many warps have their loads in flight, so the forms have
// a register cap that sets them.  Measured on GB300 (64 x 2^19 unless said;
// 128-thread blocks against 256: 2-3%, small batches 6%, less of a last wave
// is empty):
//  - f and g together (the twisted 32-bit form, so that each factor is
//    loaded once): 96 registers, five blocks, 83.8 us, 0.94 of the copy rate
//    (six, 80 registers and spills: 86.1; four: 84.9);
//  - otherwise one thread per sequence and column: 64-bit words 84 -> 63 us
//    at 128 x 2^16 against a loop over f and g.  (The 32-bit form's 128 only
//    bounds what the compiler takes, 127; smaller caps were not compared.)
constexpr int COLB = 128;
template <typename W, int NS, bool TWIST> __host__ __device__ constexpr bool cols_both() { return TWIST && NS == 2 && sizeof(W) == 4; }
template <typename W, bool BOTH, int RC>
__host__ __device__ constexpr int cols_fwd_regs() { return BOTH ? 96 : sizeof(W) == 4 ? 128 : RC <= 16 ? 80 : 168; }

template <typename W, int L, int LR, int NS, int SRC, bool TWIST>
__global__ void __maxnreg__((cols_fwd_regs<W, cols_both<W, NS, TWIST>(), (1 << (L - LR))>()))
    k_cols_fwd(const __grid_constant__ ColArgs<W> a)
{
    constexpr int RC = 1 << (L - LR);
    constexpr uint32_t N = 1u << L;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    constexpr bool BOTH = cols_both<W, NS, TWIST>();
    if (idx >= (BOTH ? a.npairs : NS * a.npairs) << LR) return;
    const long long seq = idx >> LR, pw = BOTH || NS == 1 ? seq : seq >> 1;
    const uint32_t col = (uint32_t)idx & ((1u << LR) - 1u);
    auto source = [&](int s) -> const W * {
        if constexpr (SRC == 1) {
            const DevDesc<W> d = a.descs[a.pair0 + pw];
            return s == 0 ? d.f : d.g;
        } else {
            return (s == 0 ? a.src0 : a.src1) + (size_t)(a.pair0 + pw) * N;
        }
    };
    if constexpr (BOTH) {
        // 32-bit words: f and g together, so that each twist factor is
        // loaded once for both
        const W *sf = source(0), *sg = source(1);
        W vf[RC], vg[RC];
#pragma unroll
        for (int k = 0; k < RC; ++k) {
            vf[k] = sf[col + ((uint32_t)k << LR)];
            vg[k] = sg[col + ((uint32_t)k << LR)];
        }
        col_fwd_levels<W, L, LR, L - LR - 1>(vf, a.tw, a.c);
        col_fwd_levels<W, L, LR, L - LR - 1>(vg, a.tw, a.c);
        W *df = a.dst0 + (size_t)pw * N, *dg = a.dst1 + (size_t)pw * N;
#pragma unroll
        for (int k = 0; k < RC; ++k) {
            const uint32_t x = col + ((uint32_t)k << LR);
            W z, zp;
            ld_pair_g<W>(a.pd + 2 * (size_t)x, z, zp);
            df[x] = csub<W>(shoup<W>(vf[k], z, zp, a.c.m), a.c.m);
            dg[x] = csub<W>(shoup<W>(vg[k], z, zp, a.c.m), a.c.m);
        }
    } else {
        const int s = NS == 1 ? 0 : (int)(seq & 1);
        const W *src = source(s);
        W *dst = (s == 0 ? a.dst0 : a.dst1) + (size_t)pw * N;
        W v[RC];
#pragma unroll
        for (int k = 0; k < RC; ++k) v[k] = src[col + ((uint32_t)k << LR)];
        col_fwd_levels<W, L, LR, L - LR - 1>(v, a.tw, a.c);
        if constexpr (TWIST) {
#pragma unroll
            for (int k = 0; k < RC; ++k) {
                W z, zp;
                ld_pair_g<W>(a.pd + 2 * (size_t)(col + ((uint32_t)k << LR)), z, zp);
                v[k] = csub<W>(shoup<W>(v[k], z, zp, a.c.m), a.c.m);
                // 64-bit words: keep the compiler from hoisting every table
                // load ahead of the products (it spills them otherwise)
                if constexpr (sizeof(W) == 8 && RC > 8)
                    if ((k & 7) == 7) asm volatile("" ::: "memory");
            }
        }
#pragma unroll
        for (int k = 0; k < RC; ++k) dst[col + ((uint32_t)k << LR)] = v[k];
    }
}

// Transposed top levels of the split path on column c (elements
// x = c + k 2^LR): node twiddles k >> (J + 1), the same for every column.
// Inputs < 2m; then the output stage: index <-x>_N, canonical residue.
// DST 0: contiguous out; 1: descriptor h.  ROW: log2 of the row length whose
// positions row_element maps (the twist form's), or 0 for rows in order.
template <typename W, int L, int LR, int DST, bool TWIST, int ROW>
__device__ __forceinline__ void cols_inv_body(const ColArgs<W> &a)
{
    constexpr int LC = L - LR, RC = 1 << LC;
    constexpr uint32_t N = 1u << L;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= a.npairs << LR) return;
    const long long pw = idx >> LR;
    const uint32_t col = (uint32_t)idx & ((1u << LR) - 1u);
    const W *src = a.dst0 + (size_t)pw * N;
    W *out;
    if constexpr (DST == 1) out = a.descs[a.pair0 + pw].h;
    else out = a.out + (size_t)(a.pair0 + pw) * N;
    W v[RC];
#pragma unroll
    for (int k = 0; k < RC; ++k) v[k] = src[col + ((uint32_t)k << LR)];
    uint32_t c = col;                                    // the column's own index
    if constexpr (ROW > 0) c = (col & ~((1u << ROW) - 1u)) | row_element<ROW>(col & ((1u << ROW) - 1u));
    if constexpr (TWIST) {
#pragma unroll
        for (int k = 0; k < RC; ++k) {
            W z, zp;
            ld_pair_g<W>(a.pd + 2 * (size_t)(c + ((uint32_t)k << LR)), z, zp);
            v[k] = shoup<W>(v[k], z, zp, a.c.m);
            if constexpr (sizeof(W) == 8 && RC > 8)
                if ((k & 7) == 7) asm volatile("" ::: "memory");
        }
    }
    colg_levels<W, LC, 0, 0, 0, TW_GLOBAL, RC>(v, 0u, a.tw, a.c);
#pragma unroll
    for (int k = 0; k < RC; ++k) {
        const uint32_t x = c + ((uint32_t)k << LR);
        out[(N - x) & (N - 1u)] = csub<W>(v[k], a.c.m);
    }
}

template <typename W, int L, int LR, int DST, bool TWIST, int ROW = 0>
__global__ void __maxnreg__(sizeof(W) == 8 ? 128 : 40) k_cols_inv(const __grid_constant__ ColArgs<W> a)
{
    cols_inv_body<W, L, LR, DST, TWIST, ROW>(a);
}

// The same for 32-bit words with five column bits: 72 registers, seven
// blocks per SM (512 x 2^16: 48.3 us; 48 registers, ten blocks: 52.4; 64: 49.8).
template <typename W, int L, int LR, int DST, bool TWIST, int ROW = 0>
__global__ void __maxnreg__(72) k_cols_inv5(const __grid_constant__ ColArgs<W> a)
{
    cols_inv_body<W, L, LR, DST, TWIST, ROW>(a);
}

// Split path with more column bits than one thread holds (L - LR > 5):
// the top bits run in k_cols_fwd / k_cols_inv with LR' = BLO + LB, and the
// middle bits [BLO, BLO + LB) in these kernels, in place in the wave's
// scratch.  Element x = lo + (k << BLO) + (hi << (BLO + LB)); the node of
// register bit J is x >> (BLO + J + 1) = (hi << (LB - J - 1)) | (k >> (J + 1)),
// so a column's twiddles depend on its top bits hi (read from the plan's
// table).  Forward: after the top bits; inverse (transposed): before them.
template <typename W, int L, int BLO, int LB, int NS, bool TWIST>
__global__ void __launch_bounds__(256) k_cols_mid_fwd(const __grid_constant__ ColArgs<W> a)
{
    constexpr int RC = 1 << LB, LO = L - LB;           // LO: bits outside the register group
    constexpr uint32_t N = 1u << L;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= a.npairs << LO) return;
    const long long pw = idx >> LO;
    const uint32_t r = (uint32_t)idx & ((1u << LO) - 1u);
    const uint32_t lo = r & ((1u << BLO) - 1u), hi = r >> BLO;
    const uint32_t base = lo + (hi << (BLO + LB));
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        W *p = (s == 0 ? a.dst0 : a.dst1) + (size_t)pw * N;
        W v[RC];
#pragma unroll
        for (int k = 0; k < RC; ++k) v[k] = p[base + ((uint32_t)k << BLO)];
        colf_levels<W, LB, 0, LB - 1, L - BLO - LB, TW_GLOBAL, RC>(v, hi << LB, a.tw, a.c);
        if constexpr (TWIST) {                        // the twist (brv over all L - BLO top bits)
            const uint32_t hbrv = __brev(hi) >> (32 - (L - BLO - LB));
#pragma unroll
            for (int k = 0; k < RC; ++k)
                v[k] = csub<W>(twist<W, L>(v[k], (brv_c32<LB>((uint32_t)k) << (L - BLO - LB)) | hbrv, lo, a, a.pwl), a.c.m);
        }
#pragma unroll
        for (int k = 0; k < RC; ++k) p[base + ((uint32_t)k << BLO)] = v[k];
    }
}

template <typename W, int L, int BLO, int LB, bool TWIST>
__global__ void __launch_bounds__(256) k_cols_mid_inv(const __grid_constant__ ColArgs<W> a)
{
    constexpr int RC = 1 << LB, LO = L - LB;
    constexpr uint32_t N = 1u << L;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= a.npairs << LO) return;
    const long long pw = idx >> LO;
    const uint32_t r = (uint32_t)idx & ((1u << LO) - 1u);
    const uint32_t lo = r & ((1u << BLO) - 1u), hi = r >> BLO;
    const uint32_t base = lo + (hi << (BLO + LB));
    W *p = a.dst0 + (size_t)pw * N;
    W v[RC];
#pragma unroll
    for (int k = 0; k < RC; ++k) v[k] = p[base + ((uint32_t)k << BLO)];
    if constexpr (TWIST) {
        const uint32_t hbrv = __brev(hi) >> (32 - (L - BLO - LB));
#pragma unroll
        for (int k = 0; k < RC; ++k)
            v[k] = twist<W, L>(v[k], (brv_c32<LB>((uint32_t)k) << (L - BLO - LB)) | hbrv, row_element<BLO>(lo), a, a.pwl);
    }
    colg_levels<W, LB, 0, 0, L - BLO - LB, TW_GLOBAL, RC>(v, hi << LB, a.tw, a.c);
#pragma unroll
    for (int k = 0; k < RC; ++k) p[base + ((uint32_t)k << BLO)] = v[k];
}

// Forward row levels of the split path (single sequence, in place in scratch).
template <typename W, int L, int LR>
__global__ void __launch_bounds__(BLOCK, 1) k_rows_fwd(const __grid_constant__ RowArgs<W> a)
{
    using G = Geo<W, LR>;
    constexpr int T = G::T, R = G::R, GPC = RowShape<W, L, LR>::GPC;
    constexpr uint32_t N = 1u << L;
    constexpr int last = G::NPASS - 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gid = threadIdx.x / T;
    const uint32_t tau = threadIdx.x % T;
    W *S = reinterpret_cast<W *>(smem_raw) + (size_t)gid * G::ROWP;
    const uint32_t b0 = G::base(0, tau);
    for (long long rho = (long long)blockIdx.x * GPC + gid; rho < a.nrows; rho += (long long)gridDim.x * GPC) {
        const long long pw = rho >> (L - LR);
        const uint32_t row = (uint32_t)rho & ((1u << (L - LR)) - 1u);
        W *p = const_cast<W *>(a.f) + (size_t)pw * N + ((size_t)row << LR);
        W v[1][R];
#pragma unroll
        for (int k = 0; k < R; ++k) v[0][k] = p[b0 + ((uint32_t)k << G::lo(0))];
        fwd_all<W, L, LR, 0, 1, TW_GLOBAL>(v, row << LR, tau, S, gid, a.tw, a.c);
        // back to the first pass's layout, where a warp's stores are contiguous
        if constexpr (last > 0) exchange<W, LR, last, 0, 1>(v, S, tau, gid);
#pragma unroll
        for (int k = 0; k < R; ++k) p[b0 + ((uint32_t)k << G::lo(0))] = v[0][k];
    }
}

// Forward rows of the split path's twist form, for the natural-order
// transforms: after the twisted column pass every row of 2^LR words is a
// whole length-2^LR tree with the uniform table (the first 2^(LR-1) entries
// of the plan's table), staged in shared memory.  In place, tree order: the
// same layout as the row-dependent rows (X(brv(k) + 2^LC brv(j)) at row k,
// position j), so the same bit-reversal gather follows.
template <typename W, int LR>
__global__ void __launch_bounds__(BLOCK, 1) k_rows_uni(const __grid_constant__ RowArgs<W> a)
{
    using G = Geo<W, LR>;
    using SH = NttShape<W, LR>;
    constexpr int T = G::T, R = G::R, GPC = SH::GPC;
    constexpr int last = G::NPASS - 1;
    constexpr uint32_t Q = (uint32_t)(16 / sizeof(W));
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gid = threadIdx.x / T;
    const uint32_t tau = threadIdx.x % T;
    W *stw = reinterpret_cast<W *>(smem_raw);
    W *S = reinterpret_cast<W *>(smem_raw + SH::rows) + (size_t)gid * G::ROWP;
    W *B = reinterpret_cast<W *>(smem_raw + SH::next) + (size_t)gid * SH::NB;
    const uint32_t b0 = G::base(0, tau);
    stage_twiddles<W>(a.tw, stw, TwBytes<W, LR>::pairs);
    const long long step = (long long)gridDim.x * GPC;
    long long rho = (long long)blockIdx.x * GPC + gid;
    auto stage = [&](long long r) { if (r < a.nrows) stage_seq<W, LR, Q>(a.f + ((size_t)r << LR), B, tau); };
    stage(rho);
    cp_async_wait();
    __syncthreads();
    W v[1][R];
    for (; rho < a.nrows; rho += step) {
        staged_forward<W, LR>(v, B, S, tau, gid, stw, a.c, [&] { stage(rho + step); });
        cp_async_wait();                                    // visible after the exchange's barriers
        // back to the first pass's layout, where a warp's stores are contiguous
        exchange<W, LR, last, 0, 1>(v, S, tau, gid);
        W *p = const_cast<W *>(a.f) + ((size_t)rho << LR);
#pragma unroll
        for (int k = 0; k < R; ++k) p[b0 + ((uint32_t)k << G::lo(0))] = v[0][k];
    }
}

// The same rows with the natural order written straight from them: a tile is
// the GPC rows k whose reversals brv(k) are consecutive (of one sequence),
// one per group; after their trees a row holds X(brv(k) + 2^LC u2) for all
// u2, so the tile is GPC consecutive words of every output run of 2^LC.
// INV counts the tile's rows by the output residue instead (t = <-u>_N), so
// that its runs are aligned too.  The factor a.c.ninv is the caller's (see
// k_bitrev_tiled).  It saves the bit-reversal pass, a read and a write of every
// word; GPC words of 4 bytes are a 32-byte sector for rows of 2^11 and half
// of one for 2^12, which L2 merges.
template <typename W, int L, int LR> struct RowsOutShape {
    using G = Geo<W, LR>;
    static constexpr int GPC = BLOCK / G::T, LC = L - LR;
    // rows lie RS words apart: GPC rows x consecutive words spread over all banks
    static constexpr int RS = G::ROWP + (int)(128 / sizeof(W)) / GPC;
    static constexpr size_t rows = TwBytes<W, LR>::v, next = rows + ((size_t)GPC * RS * sizeof(W) + 15) / 16 * 16;
    static constexpr size_t smem = next + (size_t)GPC * G::ROW * sizeof(W);
};

template <typename W, int L, int LR, bool INV>
__global__ void __launch_bounds__(BLOCK, 1) k_rows_out(const __grid_constant__ NttArgs<W> a)
{
    using G = Geo<W, LR>;
    using SH = RowsOutShape<W, L, LR>;
    constexpr int T = G::T, R = G::R, GPC = SH::GPC, LC = SH::LC;
    static_assert(GPC <= (1 << LC) && 32 % GPC == 0, "a tile lies in one sequence");
    constexpr uint32_t Q = (uint32_t)(16 / sizeof(W)), CM = (1u << LC) - 1u, RM = (1u << LR) - 1u;
    constexpr int TPS = (1 << LC) / GPC;                    // tiles per sequence
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gid = threadIdx.x / T;
    const uint32_t tau = threadIdx.x % T;
    W *stw = reinterpret_cast<W *>(smem_raw);
    W *rows = reinterpret_cast<W *>(smem_raw + SH::rows), *S = rows + (size_t)gid * SH::RS;
    W *B = reinterpret_cast<W *>(smem_raw + SH::next) + ((size_t)gid << LR);
    stage_twiddles<W>(a.tw, stw, TwBytes<W, LR>::pairs);
    const long long tiles = a.batch * TPS;
    auto stage = [&](long long tile) {
        if (tile >= tiles) return;
        const uint32_t res = (uint32_t)(tile % TPS) * GPC + gid, kap = INV ? (0u - res) & CM : res;
        stage_seq<W, LR, Q>(a.x + ((size_t)(tile / TPS) << L) + ((size_t)(__brev(kap) >> (32 - LC)) << LR), B, tau);
    };
    stage(blockIdx.x);
    cp_async_wait();
    __syncthreads();
    const uint32_t g = threadIdx.x % GPC, u0 = threadIdx.x / GPC;      // this thread's outputs: row g, u0 + i BLOCK / GPC
    W v[1][R];
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        staged_forward<W, LR>(v, B, S, tau, gid, stw, a.c, [&] { stage(tile + gridDim.x); });
        cp_async_wait();                                    // visible after the barriers below
        group_sync<T>(gid);
        scatter_reversed<W, LR>(v[0], S, tau);
        __syncthreads();
        const uint32_t res = (uint32_t)(tile % TPS) * GPC + g;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const uint32_t o = u0 + (uint32_t)i * (BLOCK / GPC);       // output run; INV: <-u>, one less but for residue 0
            v[0][i] = rows[g * SH::RS + G::pad(INV ? ((res == 0 ? 0u : RM) - o) & RM : o)];
        }
        __syncthreads();
        W *yp = a.y + ((size_t)(tile / TPS) << L) + res;
#pragma unroll
        for (int i = 0; i < R; ++i)
            yp[(size_t)(u0 + (uint32_t)i * (BLOCK / GPC)) << LC] = canon<W>(v[0][i], a.c.ninv, a.c.ninvp, a.c.m);
    }
}

// Bit-reversal gather of a split-path spectrum: y[u] = X(u) from the tree
// order (X(brv(x)) at x); INV applies <-u>_N.  The factor c.ninv is the
// caller's: N^-1 for the inverse, and what undoes the scale of the twist's
// diagonal.  Canonical outputs.  Tiled: write an index as (h, m, l) with h and
// l of 5 bits, so brv(h, m, l) = (brv l, brv m, brv h).  For one value of m
// the 32 x 32 elements u = (uh, m, ul) come from x = (brv ul, brv m, brv uh):
// a block reads them as 32 contiguous source runs (fixed brv ul), passes
// them through a padded shared tile, and writes 32 contiguous destination
// runs (fixed uh) -- both directions coalesced.  INV writes u to <-u>_N,
// which keeps every destination run contiguous (descending).
template <typename W, int L, bool INV>
__global__ void __launch_bounds__(256) k_bitrev_tiled(const W *__restrict__ src, W *__restrict__ dst, long long batch,
                                                     ModC<W> c)
{
    static_assert(L >= 10, "two 5-bit ends");
    constexpr uint32_t N = 1u << L;
    constexpr int LM = L - 10;                         // middle bits
    __shared__ W tile[32][33];
    const long long t = blockIdx.x;                    // (sequence, m)
    const long long b = t >> LM;
    const uint32_t m = (uint32_t)t & ((1u << LM) - 1u);
    const uint32_t mb = LM ? (__brev(m) >> (32 - LM)) : 0u;
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const W *s = src + (size_t)b * N;
    W *d = dst + (size_t)b * N;
    // source runs: x = (sh, mb, sl), sh = brv(ul) fixed per run, sl = lane
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t sh = wid * 4 + r;
        tile[sh][lane] = s[(sh << (L - 5)) | (mb << 5) | lane];
    }
    __syncthreads();
    // destination runs: u = (uh, m, ul), ul = lane; value at x = (brv ul, mb, brv uh)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t uh = wid * 4 + r;
        const uint32_t u = (uh << (L - 5)) | (m << 5) | lane;
        const W v = tile[__brev(lane) >> 27][__brev(uh) >> 27];
        d[INV ? ((N - u) & (N - 1u)) : u] = csub<W>(shoup<W>(v, c.ninv, c.ninvp, c.m), c.m);
    }
}

// ---------------------------------------------------- plain per-stage form

// One forward tree level over the whole batch of f and g: work = [2][batch][N].
template <typename W>
__global__ void k_plain_fwd(const W *__restrict__ f, const W *__restrict__ g, W *work, long long batch,
                            int L, int d, const W *__restrict__ tw, ModC<W> c)
{
    const long long half = 1ll << (L - 1);
    const long long total = 2 * batch * half;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long s = i / (batch * half);
        const long long r = i - s * batch * half;
        const long long pair = r >> (L - 1);
        const uint32_t beta = (uint32_t)(r & (half - 1));
        const int sh = L - 1 - d;
        const uint32_t node = beta >> sh;
        const uint32_t i0 = (node << (sh + 1)) | (beta & ((1u << sh) - 1u));
        const uint32_t i1 = i0 + (1u << sh);
        W *dst = work + ((size_t)s * batch + pair) * ((size_t)half * 2);
        W x0, x1;
        if (d == 0) {
            const W *sp = (s == 0 ? f : g) + (size_t)pair * ((size_t)half * 2);
            x0 = sp[i0]; x1 = sp[i1];
            ct_bfly_one<W>(x0, x1, c);
        } else {
            x0 = dst[i0]; x1 = dst[i1];
            const W z = tw[2 * node], zp = tw[2 * node + 1];
            ct_bfly<W>(x0, x1, z, zp, c);
        }
        dst[i0] = x0; dst[i1] = x1;
    }
}

template <typename W>
__global__ void k_plain_pointwise(W *work, long long batch, int L, ModC<W> c)
{
    const long long n = batch << L;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        work[i] = pointwise(work[i], work[n + i], c);
}

template <typename W>
__global__ void k_plain_inv(W *work, long long batch, int L, int d, const W *__restrict__ tw, ModC<W> c)
{
    const long long half = 1ll << (L - 1);
    const long long total = batch * half;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long pair = i >> (L - 1);
        const uint32_t beta = (uint32_t)(i & (half - 1));
        const int sh = L - 1 - d;
        const uint32_t node = beta >> sh;
        const uint32_t i0 = (node << (sh + 1)) | (beta & ((1u << sh) - 1u));
        const uint32_t i1 = i0 + (1u << sh);
        W *p = work + (size_t)pair * ((size_t)half * 2);
        W x0 = p[i0], x1 = p[i1];
        if (d == 0) gs_bfly_one<W>(x0, x1, c);
        else gs_bfly<W>(x0, x1, tw[2 * node], tw[2 * node + 1], c);
        p[i0] = x0; p[i1] = x1;
    }
}

template <typename W>
__global__ void k_plain_final(const W *__restrict__ work, W *h, long long batch, int L, ModC<W> c)
{
    const long long n = batch << L;
    const uint32_t N = 1u << L;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long pair = i >> L;
        const uint32_t x = (uint32_t)i & (N - 1u);
        h[(size_t)pair * N + ((N - x) & (N - 1u))] = csub<W>(work[i], c.m);
    }
}

// Words >= m in data[0 .. n).
template <typename W>
__global__ void k_check_range(const W *__restrict__ data, long long n, W m, unsigned long long *bad)
{
    unsigned long long cnt = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        cnt += data[i] >= m ? 1ull : 0ull;
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(bad, cnt);
}

}  // namespace ntt
