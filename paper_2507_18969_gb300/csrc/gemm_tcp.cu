// Persistent tcgen05 GEMM (gemm_tcp_kernel.cuh): BF16 and FP8, every
// epilogue mode.
#include "gemm_tcp_kernel.cuh"

namespace edpc {

cudaError_t launch_gemm_tcp(const TcGemm& g, cudaStream_t st) {
  return g.fp8 ? tcp::launch_tcp_t<true>(g, st) : tcp::launch_tcp_t<false>(g, st);
}

}  // namespace edpc
