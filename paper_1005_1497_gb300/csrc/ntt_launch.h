// ntt_launch.h -- host-side launchers of the kernels, one instantiation per
// word type (launch_u32.cu / launch_u64.cu).  Internal to the library.
#pragma once

#include <cuda_runtime.h>
#include "ntt_count.h"
#include "ntt_kernels.cuh"

namespace ntt {

constexpr int HOST_LMIN = 10;                  // lengths whose kernels read host memory without staging it
constexpr int CMAX = 5;                        // column bits of one pass of the split path

// log2 of the split path's row length (L > LRMax).  The column passes are
// bound by memory and the rows by arithmetic, so the twist form gives the
// columns more levels than the longest rows would leave them: five bits for
// 32-bit words, four for 64-bit ones (whose five-bit columns take 168
// registers), five where four would need the longest row, whose block fills
// an SM; never rows shorter than the column/row lengths.  Measured on GB300
// (conv_circular, 2, 3, 4, 5 column bits at most): 32-bit 512 x 2^16 322,
// 307, 299, 294 us and its ntt_forward 190, 188, 168, 157; 64-bit 128 x 2^16
// 278 (2), 259, 248, 263; 12 x 2^17 80 (2), 71, 71, 60.  The row-twiddle form
// keeps the longest rows.
template <typename W> constexpr int split_row_bits(int L, bool twisted)
{
    const int lo = Arith<W>::RB + 6, hi = LRMax<W>::v;     // the column/row lengths
    int lr = L - (sizeof(W) == 4 ? CMAX : CMAX - 1);
    if (lr >= hi) lr = L - CMAX;
    return !twisted || lr > hi ? hi : lr < lo ? lo : lr;
}

// Threads per block of the twist form's row kernel.
template <typename W> constexpr int row_block(int LR) { return LR < LRMax<W>::v ? BLOCK_HALF : BLOCK; }

// Threads per block of the exact convolution's fused kernels: half blocks for
// the column/row lengths below the longest, as for plain convolutions.
template <typename W> constexpr int exact_block(int L) { return L > Arith<W>::RB + 5 && L < LRMax<W>::v ? BLOCK_HALF : BLOCK; }

template <typename W> struct Launch {
    static constexpr int LRMAX = LRMax<W>::v;
    static constexpr int LMAX = 20;            // split path: LMAX - LRMAX column bits, in two passes above 5
    // rows transformed concurrently by one block of the row kernels
    static int rows_per_block(int LR);
    // pairs in flight per block of the whole-sequence fused kernels with
    // `block` threads per block (BLOCK, or BLOCK_HALF below LRMAX)
    static int pairs_per_block(int L, int block = BLOCK);
    // whether the whole-sequence fused kernels of length 2^L come with `block` threads
    static bool block_ok(int L, int block);
    // whole-sequence fused convolution (L <= LRMAX); src 0 = contiguous, 1 = descriptors,
    // 2 = contiguous in host memory (32-bit words, L >= HOST_LMIN)
    static cudaError_t conv_full(int L, int src, const RowArgs<W> &a, int grid, cudaStream_t st, int block = BLOCK);
    // (one source mode; instantiated in separate translation units)
    template <int SRC>
    static cudaError_t conv_full_src(int L, const RowArgs<W> &a, int grid, cudaStream_t st, int block);
    // one pair per block (k_conv_small) for the one-warp lengths (L <= RB + 5),
    // contiguous pairs; grid blocks walk the pairs
    static cudaError_t conv_small(int L, const RowArgs<W> &a, int grid, cudaStream_t st);
    static constexpr int SMALL_PER_SM = 32;    // largest grid of k_conv_small per SM (blocks of 32 to 256 threads)
    // split path pieces (LRMAX < L <= LMAX); cols_fwd / cols_inv run one or
    // two column passes
    // (twisted: the four-step twist form, see the twist in ntt_kernels.cuh)
    static cudaError_t conv_rows_split(int L, bool twisted, const RowArgs<W> &a, int grid, cudaStream_t st);
    static cudaError_t cols_fwd(int L, int ns, int src, bool twisted, const ColArgs<W> &a, cudaStream_t st);
    static cudaError_t cols_inv(int L, int dst, bool twisted, const ColArgs<W> &a, cudaStream_t st);
    static cudaError_t rows_fwd(int L, const RowArgs<W> &a, int grid, cudaStream_t st);
    // rows of the twist form for transforms: whole trees of the row length in place
    static cudaError_t rows_uni(int L, const RowArgs<W> &a, int grid, cudaStream_t st);
    // the same rows writing the natural order themselves, factor a.c.ninv:
    // rows per tile (0: not for this length), and the launch over a.batch sequences
    static int rows_out_rows(int L);
    static cudaError_t rows_out(int L, bool inv, const NttArgs<W> &a, int grid, cudaStream_t st);
    static cudaError_t bitrev_out(int L, bool inv, const W *src, W *dst, long long batch, const ModC<W> &c,
                                  cudaStream_t st);
    // natural-order transform of whole sequences (L <= LRMAX)
    static cudaError_t ntt_full(int L, bool inv, const NttArgs<W> &a, int grid, cudaStream_t st);
    // plain per-stage form
    static cudaError_t plain(int L, const W *f, const W *g, W *h, W *work, long long batch, const W *tw,
                             const ModC<W> &c, int grid, cudaStream_t st);
    static cudaError_t check_range(const W *data, long long n, W m, unsigned long long *bad, int grid,
                                   cudaStream_t st);
    // the exact convolution's fused launch (whole sequences, contiguous,
    // signed 64-bit h to e.h64): a plan of one prime from its signed 64-bit
    // inputs, or the second of two primes from its residues
    static cudaError_t conv_exact(int L, int primes, const RowArgs<W> &a, const ExactFused &e, int grid, cudaStream_t st);
    // dynamic shared memory of the whole-sequence fused kernel of length 2^L
    static size_t conv_full_smem(int L);
    // one persistent launch over a work list of whole-sequence items
    // (lmax: the longest length among the items; selects the instantiation)
    static cudaError_t conv_persistent(const PersistArgs<W> &a, int lmax, int grid, size_t smem, cudaStream_t st);
};

}  // namespace ntt
