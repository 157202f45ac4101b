// Fused convolution kernels reading and writing page-locked host memory in place, 32-bit words.
#include "launch_impl.cuh"
namespace ntt {
template cudaError_t Launch<uint32_t>::conv_full_src<2>(int, const RowArgs<uint32_t> &, int, cudaStream_t, int);
}  // namespace ntt
