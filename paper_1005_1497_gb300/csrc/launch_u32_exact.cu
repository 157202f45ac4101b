// The exact convolution's fused kernel instantiations (32-bit words).
#include "launch_impl.cuh"
namespace ntt {
template cudaError_t Launch<uint32_t>::conv_exact(int, int, const RowArgs<uint32_t> &, const ExactFused &, int, cudaStream_t);
}  // namespace ntt
