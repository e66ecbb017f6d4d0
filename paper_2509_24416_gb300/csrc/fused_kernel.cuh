// Fused W4A4 OBS linear: rotate-quant and the tcgen05 GEMM in one persistent
// kernel (the kernels; fused_linear.cu launches them, fused_conc_*.cu hold the
// concurrent form per type).
//
// Why not a per-tile prologue: quantizing a token needs the abs-max of its
// whole rotated row before any code exists, and a K step of the product
// needs permuted positions whose source columns are spread over the whole
// row.  For the paper's hidden sizes a 128-token block of rows does not fit
// in shared memory next to the operand pipeline, so each CTA cannot rotate
// only "its" A tile.  Instead rotate-quant (rq::run) writes the codes of
// token rows claimed from a grid-wide counter into the caller's workspace
// and publishes, per 128-token block, how many rows are done; the GEMM
// pipeline (gemm::pipeline) takes the codes in E4M3, so that TMA loads them
// straight into the MMA operand layout, and its TMA producer waits (acquire,
// bounded) until all rows of a tile's token block are published before
// loading that block's codes.  One launch, no host round trip, and the codes
// stay in L2 for the layer sizes of the paper's models.  Rows are claimed,
// not assigned, and rotate-quant never waits on the GEMM, so the producer's
// waits end as long as any CTA runs.
//
// Sequential form (fused_linear_kernel): every CTA first runs rotate-quant
// with all its threads (publishing each tile: proxy fence, CTA barrier,
// __threadfence, atomicAdd), then turns into a GEMM pipeline.
//
// Concurrent form (fused_concurrent_kernel; E4M3 weights, K <= 9216): the
// two run side by side.  Warps 0-5 of every CTA are the GEMM pipeline (of CTA
// pairs where tiles are wide) with four epilogue warps and four to six stages; warps 6-14 rotate and quantize token
// rows in the shared memory the GEMM leaves free, and warp 15 claims their
// tiles, loads and publishes them (rq::run's loader mode).  The GEMM of a
// token block starts as soon as its rows are published.
#pragma once

#include <type_traits>

#include "gemm_pipeline.cuh"
#include "rq_device.cuh"

namespace clq {

namespace {

using namespace gemm;

// Threads per CTA.  Sequential form: rotate-quant on all of them, then the
// GEMM pipeline on up to 448.  Concurrent form: GEMM warps 0-5 beside
// rotate-quant warps 6-15.
constexpr int FT = 512;

// Epilogue warps of the sequential form (unpack warps leave room for four).
template <bool BPACK>
constexpr int kSeqEpiWarps = BPACK ? 4 : 8;
// Its GEMM: CTA pairs (CG 2; 4608 x 3072 x 12288 190 -> 169 us, 16384 x 1152 x 9344
// 392 -> 362, 64 x 1152 x 12288 44.6 -> 40.5), single CTAs for packed weights and where
// pairs need a round more (single_cta_wins: 3129 x 12288 -> 3072 137.6 us before pairs,
// 142.5 on them, 130.2 on single CTAs; 300 x 9344 -> 10240 50.0, 60.6, 46.2).
template <bool BPACK, int CG>
using SeqCfg = Cfg<false, BPACK, BN, 1, 1, kSeqEpiWarps<BPACK>, MAX_STAGES, 0, CG>;

// Adds the rows [row0, row0 + rows) to the ready counters of the 128-token
// blocks they fall in (a tile of rows may straddle two blocks); RELEASE: each
// add is a release at GPU scope, else relaxed (the caller fences first).
template <bool RELEASE>
__device__ __forceinline__ void count_rows(uint32_t* ready, int row0, int rows) {
  int r = row0;
  const int end = row0 + rows;
  while (r < end) {
    const int mb = r / BM;
    const int stop = min(end, (mb + 1) * BM);
    const unsigned n = static_cast<unsigned>(stop - r);
    if (RELEASE)
      asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(ready + mb), "r"(n)
                   : "memory");
    else
      atomicAdd(ready + mb, n);
    r = stop;
  }
}

struct PublishRows {
  uint32_t* ready;
  rq::Team team;  // the threads that stored the rows
  // Every team thread, once its stores of the tile are issued: proxy fence,
  // team barrier, then one thread publishes (fence at GPU scope, adds).
  __device__ void operator()(int row0, int rows) const {
    fence_proxy_async_global();
    team.sync();
    if (team.rank() == 0) {
      __threadfence();
      count_rows<false>(ready, row0, rows);
    }
  }
  // Loader mode: the compute threads have fenced their stores for the async
  // proxy and signalled them on a CTA barrier this thread has waited on; a
  // release add at GPU scope makes them visible to every CTA that acquires
  // the counter.
  __device__ void release(int row0, int rows) const { count_rows<true>(ready, row0, rows); }
};

// Rotate-quant stage geometry of the fused kernel: its shared memory is sized
// for the GEMM pipeline anyway, so 32 KB stages let 512 threads cover as many
// rows per tile as they can (14 rows at K = 1152, 3 at K = 4608).
constexpr int kRqStride = 32 * 1024;
constexpr int kRqStages = 4;

// Concurrent form: GEMM warps 0-5, rotate-quant team warps 6-15 (compute
// warps 6-14, loader warp 15).
constexpr int kTeamFirst = (WARP_MMA + 1) * 32;  // 192
constexpr int kTeamThreads = FT - kTeamFirst;     // 320
constexpr int kTeamCompute = kTeamThreads - 32;   // 288
constexpr uint32_t kTeamBarrier = 2;  // 0: CTA, 2-3: team
constexpr int kConcStride = 18 * 1024;
constexpr int kConcStages = 3;
// The concurrent form's GEMM: CTA pairs for the wide tiles, which large products
// take (4608 x 12288 x 3072 136 -> 121 us, 16384 x 4608 x 1152 82 -> 73, 2048 x 4608 x
// 1152 19.9 -> 19.6), single CTAs for the narrow ones, where a pair's joint start costs
// more than its shared operands give (256 x 1152 x 1152 10.2 us, as pairs 11.2).
template <int BNT>
constexpr int kConcCG = BNT >= 192 ? 2 : 1;
// Its stages: what fits beside three rotate-quant stages.
template <int BNT>
constexpr int kConcGemmStages = BNT == 192 ? 5 : BNT == 64 ? 6 : 4;

template <int BNT>
struct Conc {
  using C = Cfg<false, false, BNT, 1, 1, 4, kConcGemmStages<BNT>, 0, kConcCG<BNT>>;
  static constexpr size_t RQ_OFF = (C::BYTES + 1023) & ~static_cast<size_t>(1023);
};

// F6 (both forms): the workspace codes and the weights are E2M3, loaded by
// 16U6 tensor maps (gemm::pipeline's F6 mode).
template <typename T, bool BPACK, int BNT, bool F6, int CG>
__global__ void __launch_bounds__(FT, 1)
    fused_linear_kernel(const __grid_constant__ CUtensorMap mapA,
                        const __grid_constant__ CUtensorMap mapB,
                        const __grid_constant__ CUtensorMap mapY, RotateQuantArgs rq, GemmArgs g,
                        uint32_t* ready, uint32_t* tile_counter, int use_tma_store) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ Barriers bars;
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  constexpr int EW = kSeqEpiWarps<BPACK>;
  setup<false, BPACK, BNT, 1, 1, EW, MAX_STAGES, 0, CG>(&bars);
  tc_fence_before();
  if (CG == 2)
    cluster_sync();
  else
    __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_slot;

  rq::run<T, -1, false, kRqStride, kRqStages>(rq, smem, tile_counter,
                                              PublishRows{ready, rq::Team()});
  __syncthreads();

  const Maps maps{&mapA, &mapB, use_tma_store ? &mapY : nullptr};
  pipeline<T, false, BPACK, BNT, 1, 1, false, EW, MAX_STAGES, F6, 0, CG>(maps, g, smem, &bars,
                                                                         tmem, ready);
  tc_fence_before();
  if (CG == 2)
    cluster_sync();
  else
    __syncthreads();
  teardown<CG>(tmem, SeqCfg<BPACK, CG>::TMEM);
}

template <typename T, int BNT, bool F6>
__global__ void __launch_bounds__(FT, 1)
    fused_concurrent_kernel(const __grid_constant__ CUtensorMap mapA,
                            const __grid_constant__ CUtensorMap mapB,
                            const __grid_constant__ CUtensorMap mapY, RotateQuantArgs rq,
                            GemmArgs g, uint32_t* ready, uint32_t* tile_counter,
                            int use_tma_store) {
  using C = typename Conc<BNT>::C;
  extern __shared__ uint8_t smem_raw[];
  __shared__ Barriers bars;
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  constexpr int CG = kConcCG<BNT>;
  setup<false, false, BNT, 1, 1, 4, kConcGemmStages<BNT>, 0, CG>(&bars);
  tc_fence_before();
  if (CG == 2)
    cluster_sync();  // the peer's barriers exist before anything arrives on them
  else
    __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_slot;

  if (static_cast<int>(threadIdx.x) >= kTeamFirst) {
    rq::Team team;
    team.first = kTeamFirst;
    team.count = kTeamThreads;
    team.bar = kTeamBarrier;
    rq::run<T, -1, false, kConcStride, kConcStages, false, false, PublishRows, true>(
        rq, smem + Conc<BNT>::RQ_OFF, tile_counter, PublishRows{ready, team}, team);
  } else {
    pdl_wait();  // the counters are zeroed, and Y is this kernel's to write
    const Maps maps{&mapA, &mapB, use_tma_store ? &mapY : nullptr, nullptr, nullptr};
    pipeline<T, false, false, BNT, 1, 1, false, 4, kConcGemmStages<BNT>, F6, 0, CG>(
        maps, g, smem, &bars, tmem, ready);
  }
  tc_fence_before();
  if (CG == 2)
    cluster_sync();  // a pair leaves together
  else
    __syncthreads();
  teardown<CG>(tmem, C::TMEM);
}

template <typename T, int BNT, bool F6>
cudaError_t launch_conc_t(const CUtensorMap& mapA, const CUtensorMap& mapB,
                          const CUtensorMap& mapY, const RotateQuantArgs& rq, const GemmArgs& g,
                          uint32_t* ready, int use_tma_store, size_t rq_bytes, int grid,
                          cudaStream_t st) {
  const size_t smem = Conc<BNT>::RQ_OFF + rq_bytes + 1024;  // + alignment slack
  if (smem > 227u * 1024u - 2048u) return cudaErrorInvalidValue;
  uint32_t* tile_counter = ready + (g.M + BM - 1) / BM;
  auto k = fused_concurrent_kernel<T, BNT, F6>;
  cudaError_t e = kernel_setup(reinterpret_cast<const void*>(k), smem, FT, nullptr);
  if (e != cudaSuccess) return e;
  return launch_cluster_pdl(k, grid, kConcCG<BNT>, FT, smem, st, mapA, mapB, mapY, rq, g, ready,
                            tile_counter, use_tma_store);
}

template <typename T>
cudaError_t launch_conc(const CUtensorMap& mapA, const CUtensorMap& mapB, const CUtensorMap& mapY,
                        const RotateQuantArgs& rq, const GemmArgs& g, int bn, bool f6,
                        uint32_t* ready, int use_tma_store, size_t rq_bytes, int grid,
                        cudaStream_t st) {
#define CLQ_GO(BNT, F6)                                                                         \
  return launch_conc_t<T, BNT, F6>(mapA, mapB, mapY, rq, g, ready, use_tma_store, rq_bytes, grid, st)
  switch (bn) {
    case 64:
      if (f6) CLQ_GO(64, true);
      CLQ_GO(64, false);
    case 128:
      if (f6) CLQ_GO(128, true);
      CLQ_GO(128, false);
    case 192:
      if (f6) CLQ_GO(192, true);
      CLQ_GO(192, false);
    default:
      if (f6) CLQ_GO(256, true);
      CLQ_GO(256, false);
  }
#undef CLQ_GO
}

template <typename T, bool BPACK, int BNT, bool F6, int CG>
cudaError_t launch_t(const CUtensorMap& mapA, const CUtensorMap& mapB, const CUtensorMap& mapY,
                     const RotateQuantArgs& rq, const GemmArgs& g, uint32_t* ready,
                     int use_tma_store, size_t smem, int grid, cudaStream_t st) {
  uint32_t* tile_counter = ready + (g.M + BM - 1) / BM;
  auto k = fused_linear_kernel<T, BPACK, BNT, F6, CG>;
  cudaError_t e = kernel_setup(reinterpret_cast<const void*>(k), smem, FT, nullptr);
  if (e != cudaSuccess) return e;
  return launch_cluster_pdl(k, grid, CG, FT, smem, st, mapA, mapB, mapY, rq, g, ready, tile_counter,
                            use_tma_store);
}

}  // namespace
}  // namespace clq
