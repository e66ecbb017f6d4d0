// Host side of the fused W4A4 OBS linear layer (fused_kernel.cuh): workspace
// layout, tile shapes, counters and launches.
#include "fused_kernel.cuh"
#include "fused_launch.h"

namespace clq {

namespace {

// Zeroes the readiness counters and the tile counter of a call.  A kernel rather
// than a memset, so that the fused kernel behind it may be launched with
// programmatic overlap: its barriers, tensor memory and gather offsets are set up
// while this one runs (a launch behind a memset waits for it to drain first).
__global__ void zero_counters_kernel(uint32_t* ready, int n) {
  pdl_wait();
  pdl_launch_dependents();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    ready[i] = 0u;
}

cudaError_t launch_zero_counters(uint32_t* ready, int n, cudaStream_t st) {
  return launch_pdl(zero_counters_kernel, std::min((n + 255) / 256, 64), 256, 0, st, ready, n);
}

size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

}  // namespace

FusedWorkspace fused_workspace_layout(int M, int K) {
  FusedWorkspace w{};
  const size_t m = static_cast<size_t>(M < 0 ? 0 : M);
  w.codes_off = 0;
  w.scales_off = align256(m * static_cast<size_t>(K));  // E4M3 codes
  w.ready_off = align256(w.scales_off + 4 * m);
  w.bytes = align256(w.ready_off + 4 * ((m + BM - 1) / BM + 1));  // + tile counter
  return w;
}

namespace {

// Concurrent form (E4M3 weights): rows per tile as the 288 compute threads
// and a 18 KB stage allow (8 at K = 1152, 2 at K = 4608).
cudaError_t launch_concurrent(const RotateQuantArgs& rq_in, const uint8_t* W, int w_codes,
                              const GemmArgs& g, int logb, int dtype, uint32_t* ready, int sms,
                              cudaStream_t st) {
  RotateQuantArgs rq = rq_in;
  rq.logb = logb;
  const bool f6 = w_codes == CLQ_CODES_E2M3;
  const int a_codes = f6 ? CLQ_CODES_E2M3 : CLQ_CODES_E4M3;  // the weights' family
  rq.e4m3 = f6 ? 3 : 1;
  const int segs = rq.K / 32;
  const int R = std::min(kTeamCompute / segs, kConcStride / (2 * rq.K));
  if (R < 1) return cudaErrorInvalidValue;
  rq.rows_per_tile = R;
  // The narrow tiles' gain, us: 256 x 1152 x 1152 12.9 -> 10.5, 875 x 5120 x 192 32.1 ->
  // 23.7, 1024 x 1152 x 1152 13.4 -> 11.4.
  int bn = gemm_tile_n(g.M, g.N, g.K, BM, sms, true, true, 1100);
  const int cg = bn >= 192 ? 2 : 1;  // CTA pairs (kConcCG)
  if (cg == 2) bn = gemm_tile_n(g.M, g.N, g.K, 2 * BM, sms / 2, true, false, 1100);
  const size_t rq_bytes = rq::smem_bytes(R, kConcStride, kConcStages);

  const int tiles_m = (g.M + BM - 1) / BM;
  cudaError_t e = launch_zero_counters(ready, tiles_m + 1, st);
  if (e != cudaSuccess) return e;
  CUtensorMap mapA, mapB, mapY;
  if (!encode_codes_map(&mapA, rq.Q, a_codes, g.M, g.K, BM, 0) ||
      !encode_codes_map(&mapB, W, w_codes, g.N, g.K, bn / cg, 0))
    return cudaErrorInvalidValue;
  const int use_tma_store = (g.N % 8 == 0) ? 1 : 0;
  if (use_tma_store) {
    if (!encode_tma_out_tile(&mapY, g.Y, g.M, g.N)) return cudaErrorInvalidValue;
  } else {
    mapY = mapA;  // unused
  }
  auto* go = dtype == CLQ_F16 ? launch_conc_f16 : launch_conc_bf16;
  return go(mapA, mapB, mapY, rq, g, bn, f6, ready, use_tma_store, rq_bytes, sms / cg * cg, st);
}

}  // namespace

cudaError_t launch_fused_linear(const RotateQuantArgs& rq_in, const uint8_t* W, int w_codes,
                                const GemmArgs& g, int logb, int dtype, uint32_t* ready,
                                cudaStream_t st) {
  const bool bpack = w_codes == CLQ_CODES_INT4_PACKED;
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  if (!bpack && rq_in.K <= kConcStride / 2 && rq_in.K / 32 <= kTeamCompute)
    return launch_concurrent(rq_in, W, w_codes, g, logb, dtype, ready, sms, st);
  const int bn = BN;
  const int cg = bpack || single_cta_wins(g.M, g.N, g.K, 1, bn, sms, false) ? 1 : 2;
  const size_t gemm_bytes = bpack     ? SeqCfg<true, 1>::BYTES
                            : cg == 1 ? SeqCfg<false, 1>::BYTES
                                      : SeqCfg<false, 2>::BYTES;
  const size_t limit = 227u * 1024u - 2048u;  // dynamic + static shared memory
  // Rotate-quant phase: as many rows per tile as 512 threads cover and one
  // raw stage holds.
  RotateQuantArgs rq = rq_in;
  rq.logb = logb;
  // the workspace holds the codes in the GEMM's operand layout: E2M3 beside
  // E2M3 weights, else E4M3
  const bool f6 = w_codes == CLQ_CODES_E2M3;
  rq.e4m3 = f6 ? 3 : 1;
  const int segs = rq.K / 32;
  const int R = std::max(1, std::min(FT / segs, kRqStride / (2 * rq.K)));
  const size_t rq_bytes = rq::smem_bytes(R, kRqStride, kRqStages);
  if (rq_bytes > limit || R * segs > FT) return cudaErrorInvalidValue;
  rq.rows_per_tile = R;
  const size_t smem = std::max(gemm_bytes, rq_bytes) + 1024;

  const int tiles_m = (g.M + BM - 1) / BM;
  cudaError_t e = launch_zero_counters(ready, tiles_m + 1, st);
  if (e != cudaSuccess) return e;

  CUtensorMap mapA, mapB, mapY;
  if (!encode_codes_map(&mapA, rq.Q, f6 ? CLQ_CODES_E2M3 : CLQ_CODES_E4M3, g.M, g.K, BM, 0) ||
      !encode_codes_map(&mapB, W, w_codes, g.N, g.K, bn / cg, 0))
    return cudaErrorInvalidValue;
  const int use_tma_store = (g.N % 8 == 0) ? 1 : 0;
  if (use_tma_store) {
    if (!encode_tma_out_tile(&mapY, g.Y, g.M, g.N)) return cudaErrorInvalidValue;
  } else {
    mapY = mapA;  // unused
  }
  const int grid = sms / cg * cg;
#define CLQ_GO(BPACK, F6, CG)                                                                    \
  return dtype == CLQ_F16                                                                        \
             ? launch_t<__half, BPACK, BN, F6, CG>(mapA, mapB, mapY, rq, g, ready,               \
                                                   use_tma_store, smem, grid, st)                \
             : launch_t<__nv_bfloat16, BPACK, BN, F6, CG>(mapA, mapB, mapY, rq, g, ready,        \
                                                          use_tma_store, smem, grid, st)
  if (bpack) CLQ_GO(true, false, 1);
  if (f6 && cg == 1) CLQ_GO(false, true, 1);
  if (f6) CLQ_GO(false, true, 2);
  if (cg == 1) CLQ_GO(false, false, 1);
  CLQ_GO(false, false, 2);
#undef CLQ_GO
}

}  // namespace clq
