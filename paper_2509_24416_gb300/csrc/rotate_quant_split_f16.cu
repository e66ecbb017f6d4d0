// Hot-path rotate-quantize kernel variants (wide segments, b >= 64): __half input,
// 8-bit codes in split planes.
#include "rq_launch.cuh"

namespace clq {

cudaError_t launch_rotate_quant_wide_f16_split(const RotateQuantArgs& a, int logb, int stage,
                                              int threads, size_t smem, int sms,
                                              cudaStream_t st) {
  return rq::launch_rotate_quant_wide_t<__half, 2>(a, logb, stage, threads, smem, sms, st);
}

}  // namespace clq
