// Interface between the GEMM's host side (w4a4_gemm.cu) and its kernels, compiled
// once per output type.
#pragma once

#include "clq_kernels.h"

namespace clq {

// Largest K for which W8A8's cross and low products share one exact fp32
// accumulator: at most 2112 a code pair (gemm_pipeline.cuh), 2112 K < 2^24.
constexpr int kSep2MaxK = 7936;

// Tensor maps of a launch: operands, output, second planes of 8-bit operands.
struct MapSet {
  CUtensorMap A, B, Y, A2, B2;
};

// Tile shape of a launch: cg * 128 rows (a CTA or a CTA pair) x bn columns (pairs, for
// execution-layout operands: 256, 192, 128 or 64, W8A8 128 or 64; single CTAs, for
// those too and for packed ones: 256, W8A8 128).
struct TileShape {
  int cg, bn;
};

// One launcher per operand family and output type, each in its own translation
// unit (gemm_*.cu) so that they compile in parallel:
//   e4m3: E4M3 x E4M3, symmetric
//   e2m3: E2M3 x E2M3
//   bits: 8-bit (split) activations, symmetric or asymmetric, and asymmetric 4-bit E4M3
//   packed: packed nibbles on either side
cudaError_t launch_gemm_e4m3_f16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                 TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_e4m3_bf16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                  TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_e2m3_f16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                 TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_e2m3_bf16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                  TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_bits_f16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                 TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_bits_bf16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                  TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_packed_f16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                   TileShape t, int use_tma_store, int grid, cudaStream_t st);
cudaError_t launch_gemm_packed_bf16(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                                    TileShape t, int use_tma_store, int grid, cudaStream_t st);

}  // namespace clq
