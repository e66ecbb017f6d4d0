// GEMM kernels: 8-bit (split) activations, symmetric or asymmetric, and asymmetric 4-bit E4M3; bf16 outputs.
#include "gemm_kernel.cuh"

namespace clq {

cudaError_t launch_gemm_bits_bf16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                  TileShape t, int use_tma_store, int grid, cudaStream_t st) {
  return launch_gemm_bits<__nv_bfloat16>(m, g, x_codes, w_codes, t, use_tma_store, grid, st);
}

}  // namespace clq
