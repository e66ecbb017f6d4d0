// Concurrent fused kernels, __half.
#include "fused_kernel.cuh"
#include "fused_launch.h"

namespace clq {

cudaError_t launch_conc_f16(const CUtensorMap& mapA, const CUtensorMap& mapB,
                            const CUtensorMap& mapY, const RotateQuantArgs& rq, const GemmArgs& g,
                            int bn, bool f6, uint32_t* ready, int use_tma_store, size_t rq_bytes,
                            int grid, cudaStream_t st) {
  return launch_conc<__half>(mapA, mapB, mapY, rq, g, bn, f6, ready, use_tma_store, rq_bytes, grid,
                         st);
}

}  // namespace clq
