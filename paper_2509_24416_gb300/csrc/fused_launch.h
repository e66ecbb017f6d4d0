// Interface between the fused layer's host side (fused_linear.cu) and the
// concurrent form's kernels, compiled once per type.
#pragma once

#include "clq_kernels.h"

namespace clq {

// bn: tile columns (256, 192, 128 or 64); f6: E2M3 codes; rq_bytes: shared memory
// of the rotate-quant team.
cudaError_t launch_conc_f16(const CUtensorMap& mapA, const CUtensorMap& mapB,
                            const CUtensorMap& mapY, const RotateQuantArgs& rq, const GemmArgs& g,
                            int bn, bool f6, uint32_t* ready, int use_tma_store, size_t rq_bytes,
                            int grid, cudaStream_t st);
cudaError_t launch_conc_bf16(const CUtensorMap& mapA, const CUtensorMap& mapB,
                             const CUtensorMap& mapY, const RotateQuantArgs& rq,
                             const GemmArgs& g, int bn, bool f6, uint32_t* ready,
                             int use_tma_store, size_t rq_bytes, int grid, cudaStream_t st);

}  // namespace clq
