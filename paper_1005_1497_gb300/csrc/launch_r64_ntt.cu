// Natural-order transform kernels for 64-bit words of moduli below 2^48 (r64).
#include "launch_impl.cuh"
namespace ntt {
template cudaError_t Launch<r64>::ntt_full(int, bool, const NttArgs<r64> &, int, cudaStream_t);
template cudaError_t Launch<r64>::rows_uni(int, const RowArgs<r64> &, int, cudaStream_t);
template cudaError_t Launch<r64>::rows_out(int, bool, const NttArgs<r64> &, int, cudaStream_t);
}  // namespace ntt
