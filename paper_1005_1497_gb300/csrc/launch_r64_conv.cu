// Fused convolution kernels on contiguous batches and split-path rows for 64-bit words of moduli below 2^48 (r64).
#include "launch_impl.cuh"
namespace ntt {
template cudaError_t Launch<r64>::conv_full_src<0>(int, const RowArgs<r64> &, int, cudaStream_t, int);
template cudaError_t Launch<r64>::conv_rows_split(int, bool, const RowArgs<r64> &, int, cudaStream_t);
}  // namespace ntt
