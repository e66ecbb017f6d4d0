// Interface between the GEMM's host side (w4a4_gemm.cu) and its kernels, compiled
// once per output type.
#pragma once

#include "clq_kernels.h"

namespace clq {

// W8A8 tiles: three accumulators of 128 columns fill one TMEM allocation.
constexpr int kSepBN = 128;

// Tensor maps of a launch: operands, output, second planes of 8-bit operands.
struct MapSet {
  CUtensorMap A, B, Y, A2, B2;
};

// Tile shape of a launch: cg * 128 rows (a CTA or a CTA pair) x bn columns.
struct TileShape {
  int cg, bn;
};

cudaError_t launch_gemm_f16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                            TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_bf16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                             TileShape t, int use_tma_store, int grid, cudaStream_t st);

}  // namespace clq
