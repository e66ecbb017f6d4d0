// Standalone GEMM kernel around gemm::pipeline and its launch for every operand
// layout and tile shape; included once per operand family and output type so that
// the variants compile in parallel.
#pragma once

#include "gemm_launch.h"
#include "gemm_pipeline.cuh"

namespace clq {
namespace {

using namespace gemm;

template <bool APACK, bool BPACK, int BNT, int PA, int PB, int SEP, int CG>
using KernelCfg = Cfg<APACK, BPACK, BNT, PA, PB, 0, MAX_STAGES, SEP, CG>;

// PA / PB = 2: the activation / weight codes are 8-bit, as two E4M3 planes
// (mapA2 / mapB2 the second plane).  CG 2: launched as clusters of two CTAs,
// each pair sharing 256 x BNT tiles (tcgen05 cta_group::2).
template <typename OutT, bool APACK, bool BPACK, int BNT, int PA, int PB, bool ASYM, bool F6,
          int SEP, int CG>
__global__ void __launch_bounds__((KernelCfg<APACK, BPACK, BNT, PA, PB, SEP, CG>::THREADS), 1)
    w4a4_gemm_kernel(const __grid_constant__ CUtensorMap mapA,
                     const __grid_constant__ CUtensorMap mapB,
                     const __grid_constant__ CUtensorMap mapY,
                     const __grid_constant__ CUtensorMap mapA2,
                     const __grid_constant__ CUtensorMap mapB2, GemmArgs g, int use_tma_store) {
  using C = KernelCfg<APACK, BPACK, BNT, PA, PB, SEP, CG>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ Barriers bars;
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  setup<APACK, BPACK, BNT, PA, PB, 0, MAX_STAGES, SEP, CG>(&bars);
  tc_fence_before();
  if (CG == 2)
    cluster_sync();  // the peer's barriers exist before anything arrives on them
  else
    __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_slot;
  // The tensor maps are kernel parameters, not outputs of the previous kernel:
  // fetch them while it finishes (measured +0.25 % on the PixArt step).
  if (threadIdx.x == WARP_TMA * 32) {
    prefetch_tensor_map(&mapA);
    prefetch_tensor_map(&mapB);
    if (use_tma_store) prefetch_tensor_map(&mapY);
    // The weight boxes of this CTA's first pipeline stages into L2 (a hint:
    // it changes no value the copies after the wait read).
    constexpr int TM = CG * BM;
    const int tiles_n = (g.N + BNT - 1) / BNT;
    const int tiles = ((g.M + TM - 1) / TM) * tiles_n;
    const int unit = static_cast<int>(blockIdx.x) / CG;
    if (!BPACK && unit < tiles) {
      const int rank = CG == 2 ? static_cast<int>(cluster_ctarank()) : 0;
      const int n0 = (unit % tiles_n) * BNT + rank * (BNT / CG);
      const int nk = (g.K + BK - 1) / BK;
      for (int kb = 0; kb < C::S && kb < nk; ++kb) {
        tma_prefetch_2d(&mapB, kb * BK, n0);
        if (PB == 2) tma_prefetch_2d(&mapB2, kb * BK, n0);
      }
    }
  }
  // Barriers and TMEM are set up; global inputs are read only from here on.
  pdl_wait();
  pdl_launch_dependents();
  const Maps maps{&mapA, &mapB, use_tma_store ? &mapY : nullptr, &mapA2, &mapB2};
  pipeline<OutT, APACK, BPACK, BNT, PA, PB, ASYM, 0, MAX_STAGES, F6, SEP, CG>(maps, g, smem, &bars,
                                                                              tmem, nullptr);
  tc_fence_before();
  // A pair leaves together: either CTA's barriers and shared memory may be
  // written by the other until then.
  if (CG == 2)
    cluster_sync();
  else
    __syncthreads();
  teardown<CG>(tmem, C::TMEM);
}

template <typename OutT, bool APACK, bool BPACK, int BNT, int CG = 1, int PA = 1, int PB = 1,
          bool ASYM = false, bool F6 = false, int SEP = 0>
cudaError_t launch_gemm_t(const MapSet& m, const GemmArgs& g, int use_tma_store, int grid,
                          cudaStream_t st) {
  using C = KernelCfg<APACK, BPACK, BNT, PA, PB, SEP, CG>;
  auto k = w4a4_gemm_kernel<OutT, APACK, BPACK, BNT, PA, PB, ASYM, F6, SEP, CG>;
  constexpr size_t smem = C::BYTES + 1024;  // + alignment slack
  cudaError_t e = kernel_setup(reinterpret_cast<const void*>(k), smem, C::THREADS, nullptr);
  if (e != cudaSuccess) return e;
  return launch_cluster_pdl(k, grid, CG, C::THREADS, smem, st, m.A, m.B, m.Y, m.A2, m.B2, g,
                            use_tma_store);
}

// CTA pairs for operands in an execution layout, single CTAs for packed ones (whose
// unpack warps work on a whole tile's operands) and for the widest tile where
// single_cta_wins.
#define CLQ_GO(...) return launch_gemm_t<OutT, __VA_ARGS__>(m, g, use_tma_store, grid, st)

template <typename OutT>
cudaError_t launch_gemm_e4m3(const MapSet& m, const GemmArgs& g, int, int, TileShape t,
                             int use_tma_store, int grid, cudaStream_t st) {
  if (t.cg == 1) CLQ_GO(false, false, 256, 1);
  switch (t.bn) {
    case 64: CLQ_GO(false, false, 64, 2);
    case 128: CLQ_GO(false, false, 128, 2);
    case 192: CLQ_GO(false, false, 192, 2);
    default: CLQ_GO(false, false, 256, 2);
  }
}

template <typename OutT>
cudaError_t launch_gemm_e2m3(const MapSet& m, const GemmArgs& g, int, int, TileShape t,
                             int use_tma_store, int grid, cudaStream_t st) {
  if (t.cg == 1) CLQ_GO(false, false, 256, 1, 1, 1, false, true);
  switch (t.bn) {
    case 64: CLQ_GO(false, false, 64, 2, 1, 1, false, true);
    case 128: CLQ_GO(false, false, 128, 2, 1, 1, false, true);
    case 192: CLQ_GO(false, false, 192, 2, 1, 1, false, true);
    default: CLQ_GO(false, false, 256, 2, 1, 1, false, true);
  }
}

template <typename OutT>
cudaError_t launch_gemm_bits(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                             TileShape t, int use_tma_store, int grid, cudaStream_t st) {
  const bool a8 = x_codes == CLQ_CODES_E4M3_SPLIT, w8 = w_codes == CLQ_CODES_E4M3_SPLIT;
  if (t.cg == 1) {
    if (g.lo != nullptr) {
      if (a8 && w8 && g.K > kSep2MaxK) CLQ_GO(false, false, 128, 1, 2, 2, true, false, 3);
      if (a8 && w8) CLQ_GO(false, false, 128, 1, 2, 2, true, false, 2);
      if (a8) CLQ_GO(false, false, 256, 1, 2, 1, true);
      CLQ_GO(false, false, 256, 1, 1, 1, true);
    }
    if (w8 && g.K > kSep2MaxK) CLQ_GO(false, false, 128, 1, 2, 2, false, false, 3);
    if (w8) CLQ_GO(false, false, 128, 1, 2, 2, false, false, 2);
    CLQ_GO(false, false, 256, 1, 2, 1);
  }
  if (g.lo != nullptr) {  // asymmetric activations
    if (a8 && w8 && g.K > kSep2MaxK) CLQ_GO(false, false, 128, 2, 2, 2, true, false, 3);
    if (a8 && w8) CLQ_GO(false, false, 128, 2, 2, 2, true, false, 2);
    if (a8) CLQ_GO(false, false, 256, 2, 2, 1, true);
    switch (t.bn) {
      case 64: CLQ_GO(false, false, 64, 2, 1, 1, true);
      case 128: CLQ_GO(false, false, 128, 2, 1, 1, true);
      default: CLQ_GO(false, false, 256, 2, 1, 1, true);
    }
  }
  if (w8 && g.K > kSep2MaxK) CLQ_GO(false, false, 128, 2, 2, 2, false, false, 3);
  if (w8 && t.bn == 64) CLQ_GO(false, false, 64, 2, 2, 2, false, false, 2);
  if (w8) CLQ_GO(false, false, 128, 2, 2, 2, false, false, 2);
  switch (t.bn) {
    case 64: CLQ_GO(false, false, 64, 2, 2, 1);
    case 128: CLQ_GO(false, false, 128, 2, 2, 1);
    default: CLQ_GO(false, false, 256, 2, 2, 1);
  }
}

template <typename OutT>
cudaError_t launch_gemm_packed(const MapSet& m, const GemmArgs& g, int x_codes, int w_codes,
                               TileShape, int use_tma_store, int grid, cudaStream_t st) {
  const bool apack = x_codes == CLQ_CODES_INT4_PACKED;
  const bool bpack = w_codes == CLQ_CODES_INT4_PACKED;
  if (apack && bpack) CLQ_GO(true, true, BN);
  if (apack) CLQ_GO(true, false, BN);
  CLQ_GO(false, true, BN);
}
#undef CLQ_GO

}  // namespace
}  // namespace clq
