// GEMM kernels: E4M3 x E4M3, symmetric; f16 outputs.
#include "gemm_kernel.cuh"

namespace clq {

cudaError_t launch_gemm_e4m3_f16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                 TileShape t, int use_tma_store, int grid, cudaStream_t st) {
  return launch_gemm_e4m3<__half>(m, g, x_codes, w_codes, t, use_tma_store, grid, st);
}

}  // namespace clq
