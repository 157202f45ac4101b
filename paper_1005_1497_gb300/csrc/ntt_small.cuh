// ntt_small.cuh -- the whole convolution of one short pair by one thread
// block, for batches too small to fill the GPU with the kernels that give
// each pair one warp (k_conv_fused).
//
// The block form of ntt_block.cuh: forward levels D = 0 .. L - BB - 1, node i
// of level D pairing the elements at distance 2^{L-1-D} with the twiddle z_i
// (the plan's table), products modulo x^4 -+ z_i, decimation-in-time inverse
// of the four subsequences, last factor and output index as there; lengths
// below 8 are convolved directly.
//
// A single pair is bound by latency: a chain of steps, each a round trip
// through shared memory and a block barrier.  So a step holds three levels
// (eight elements per work item; two for 64-bit words, whose longer code and
// register use cost more than the barriers saved), the first step reads the
// inputs and its few twiddles straight from device memory while the table is
// on its way, the last one writes the output, and the block has the threads
// that fill the steps: 2^10 takes six barriers.  Measured on GB300 in a
// graph of launches, the complete transform by two levels a step with 256
// threads against this form (bit-identical): 1 x 2^10 4.53 -> 2.55 us, 608 x
// 2^10 8.25 -> 5.07, 2432 x 2^8 7.23 -> 4.66, 1 x 2^6 1.96 -> 1.92; 64-bit
// words 1 x 2^9 4.56 -> 3.29, 608 x 2^8 5.60 -> 4.42 (by three levels a step
// and half the threads 3.60 and 4.64).  The one-warp kernels win once the
// batch fills the GPU, which decides the plan's small-batch limit.
#pragma once
#include "ntt_block.cuh"
#include "ntt_kernels.cuh"

namespace ntt {

template <typename W, int L> struct SmallShape {
    static constexpr uint32_t N = 1u << L;
    static constexpr bool BLOCKS = L >= BLOCK_LMIN;
    static constexpr int LV = BLOCKS ? L - BB : 0;               // levels
    static constexpr int KMAX = sizeof(W) == 4 ? 3 : 2;          // levels of a step
    static constexpr int KE = LV < KMAX ? LV : KMAX;             // of the first and the last one
    // threads: an item each of the widest step, one warp at least
    static constexpr int TL = L - KMAX + 1;
    static constexpr int THREADS = TL <= 5 ? 32 : 1 << TL;
    static constexpr int PER_SM = (sizeof(W) == 4 ? 1024 : 512) / THREADS;   // 64 or 128 registers
    // Four pad words every 32 (64-bit words: 16): all steps' accesses and the
    // products' aligned groups of four are free of bank conflicts.
    __host__ __device__ static constexpr uint32_t pad(uint32_t x) { return x + 4 * (x >> Arith<W>::PADSH); }
    static constexpr uint32_t ROWA = (pad(N - 1) + 4u) & ~3u;    // words of one sequence's region
    static constexpr uint32_t TWP = BLOCKS ? N / (2u << BB) : 0; // (twiddle, quotient) pairs of the table
    static constexpr size_t smem = (2 * (size_t)ROWA + 2 * (size_t)TWP) * sizeof(W);
    // levels of the next step when r remain besides the first or the last one's
    __host__ __device__ static constexpr int middle(int r) { return r == 4 ? 2 : (r < KMAX ? r : KMAX); }
};

// Levels D .. D + K - 1 of the 2^K elements v of one item in node i of level
// D.  tw: any table of (twiddle, quotient) pairs.
template <typename W, int D, int K>
__device__ __forceinline__ void small_fwd_levels(W (&v)[1 << K], uint32_t i, const W *__restrict__ tw, const ModC<W> &c)
{
#pragma unroll
    for (int s = 0; s < K; ++s) {
        const int h = 1 << (K - 1 - s);
#pragma unroll
        for (int n = 0; n < (1 << s); ++n) {
            if (D + s == 0) {
#pragma unroll
                for (int j = 0; j < h; ++j) ct_bfly_one<W>(v[j], v[j + h], c);
                continue;
            }
            const uint32_t e = 2u * ((i << s) + (uint32_t)n);
            const W z = tw[e], zp = tw[e + 1];
#pragma unroll
            for (int j = 0; j < h; ++j) ct_bfly<W>(v[2 * n * h + j], v[2 * n * h + j + h], z, zp, c);
        }
    }
}

// Inverse levels l .. l + K - 1 (element bits BB + l ..) of the 2^K elements
// v of one item whose block index has the low l bits brv(t).
template <typename W, int l, int K>
__device__ __forceinline__ void small_inv_levels(W (&v)[1 << K], uint32_t t, const W *__restrict__ tw, const ModC<W> &c)
{
#pragma unroll
    for (int J = 0; J < K; ++J)
#pragma unroll
        for (int n = 0; n < (1 << J); ++n) {
            const int low = J == 0 ? 0 : (J == 1 ? n : (int)brv_c<2>(n));
            if (l + J == 0) {
#pragma unroll
                for (int k = 0; k < (1 << K); k += 2) ct_bfly_unit<W>(v[k], v[k + 1], 23 * c.m);
                continue;
            }
            const uint32_t e = 2u * ((t << J) + (uint32_t)n);
            const W z = tw[e], zp = tw[e + 1];
#pragma unroll
            for (int hi = 0; hi < (1 << K); hi += 2 << J) ct_bfly<W>(v[hi | low], v[hi | low | 1 << J], z, zp, c);
        }
}

// Forward levels D, D + 1, ... of f and g in shared memory, after the first step.
template <typename W, int L, int D>
__device__ __forceinline__ void small_fwd(W *S, const W *zt, const ModC<W> &c)
{
    using SH = SmallShape<W, L>;
    if constexpr (D < SH::LV) {
        constexpr int K = SH::middle(SH::LV - D);
        constexpr uint32_t q = SH::N >> (D + K), items = SH::N >> K;
        for (uint32_t u = threadIdx.x; u < 2 * items; u += SH::THREADS) {
            const uint32_t w = u & (items - 1), i = w / q;
            W *x = S + (u < items ? 0u : SH::ROWA);
            const uint32_t p = i * (q << K) + w % q;
            W v[1 << K];
#pragma unroll
            for (int k = 0; k < (1 << K); ++k) v[k] = x[SH::pad(p + k * q)];
            small_fwd_levels<W, D, K>(v, i, zt, c);
#pragma unroll
            for (int k = 0; k < (1 << K); ++k) x[SH::pad(p + k * q)] = v[k];
        }
        __syncthreads();
        small_fwd<W, L, D + K>(S, zt, c);
    }
}

// Inverse levels l, l + 1, ... up to the last step, which writes the output.
template <typename W, int L, int l>
__device__ __forceinline__ void small_inv(W *S, W *__restrict__ h, const W *zt, const ModC<W> &c)
{
    using SH = SmallShape<W, L>;
    constexpr bool last = l == SH::LV - SH::KE;
    constexpr int K = last ? SH::KE : SH::middle(SH::LV - SH::KE - l);
    constexpr uint32_t q = 1u << (BB + l), items = SH::N >> K;
    for (uint32_t u = threadIdx.x; u < items; u += SH::THREADS) {
        const uint32_t lo = u % q, p = u / q * (q << K) + lo;
        W v[1 << K];
#pragma unroll
        for (int k = 0; k < (1 << K); ++k) v[k] = S[SH::pad(p + k * q)];
        uint32_t t = 0;
        if constexpr (l > 0) t = __brev(lo >> BB) >> (32 - l);
        small_inv_levels<W, l, K>(v, t, zt, c);
#pragma unroll
        for (int k = 0; k < (1 << K); ++k) {
            if constexpr (last) h[block_out<L>(p + k * q)] = canon<W>(v[k], c.cB, c.cBp, c.m);
            else S[SH::pad(p + k * q)] = v[k];
        }
    }
    __syncthreads();
    if constexpr (!last) small_inv<W, L, l + K>(S, h, zt, c);
}

// Pairs blockIdx.x, blockIdx.x + gridDim.x, ... of contiguous f, g, h.
// Inputs in [0, m); outputs canonical.
template <typename W, int L>
__global__ void __launch_bounds__(SmallShape<W, L>::THREADS, SmallShape<W, L>::PER_SM) k_conv_small(const __grid_constant__ RowArgs<W> a)
{
    using SH = SmallShape<W, L>;
    constexpr uint32_t N = SH::N;
    if constexpr (!SH::BLOCKS) {
        using D = typename Wide<W>::T;
        for (long long pr = blockIdx.x; pr < a.nrows; pr += gridDim.x) {
            const size_t off = (size_t)(a.pair0 + pr) * N;
            const uint32_t t = threadIdx.x & (N - 1u);
            D s = 0;
#pragma unroll
            for (uint32_t i = 0; i < N; ++i) s += (D)a.f[off + i] * a.g[off + ((t - i) & (N - 1u))];
            const W v = shoup<W>(mont(s, a.c), a.c.cN, a.c.cNp, a.c.m) << L;         // 2^B N^{-1}, N
            __syncwarp();                                                            // h may be f or g
            if (threadIdx.x < N) a.h[off + t] = canon<W>(v, (W)1, a.c.onep, a.c.m);
        }
        return;
    } else {
        extern __shared__ __align__(16) unsigned char smem_small[];
        W *S = reinterpret_cast<W *>(smem_small), *zt = S + 2 * SH::ROWA;
        for (uint32_t i = threadIdx.x; i < 2 * SH::TWP; i += SH::THREADS) zt[i] = a.tw[i];
        for (long long pr = blockIdx.x; pr < a.nrows; pr += gridDim.x) {
            const size_t off = (size_t)(a.pair0 + pr) * N;
            constexpr int K = SH::KE;
            constexpr uint32_t q = N >> K;
            for (uint32_t u = threadIdx.x; u < 2 * q; u += SH::THREADS) {
                const uint32_t j = u & (q - 1);
                const W *in = (u < q ? a.f : a.g) + off + j;
                W *x = S + (u < q ? 0u : SH::ROWA);
                W v[1 << K];
#pragma unroll
                for (int k = 0; k < (1 << K); ++k) v[k] = in[k * q];
                small_fwd_levels<W, 0, K>(v, 0u, a.tw, a.c);
#pragma unroll
                for (int k = 0; k < (1 << K); ++k) x[SH::pad(j + k * q)] = v[k];
            }
            __syncthreads();
            small_fwd<W, L, K>(S, zt, a.c);
            for (uint32_t u = threadIdx.x; u < N >> BB; u += SH::THREADS) {
                W *x = S + SH::pad(u << BB);
                W v[2][1 << BB];
                ld_vec<W, 1 << BB>(x, v[0], true);
                ld_vec<W, 1 << BB>(x + SH::ROWA, v[1], true);
                block_product<W, 1 << BB>(v, 0, u & 1u, zt[u & ~1u], zt[u | 1u], a.c);
                st_vec<W, 1 << BB>(x, v[0], true);
            }
            __syncthreads();
            small_inv<W, L, 0>(S, a.h + off, zt, a.c);
        }
    }
}

}  // namespace ntt
