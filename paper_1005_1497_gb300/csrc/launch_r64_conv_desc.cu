// Fused convolution kernels on descriptor lists for 64-bit words of moduli below 2^48 (r64).
#include "launch_impl.cuh"
namespace ntt {
template bool Launch<r64>::block_ok(int, int);
template cudaError_t Launch<r64>::conv_full(int, int, const RowArgs<r64> &, int, cudaStream_t, int);
template cudaError_t Launch<r64>::conv_full_src<1>(int, const RowArgs<r64> &, int, cudaStream_t, int);
}  // namespace ntt
