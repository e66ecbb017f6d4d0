// Hot-path rotate-quantize kernel variants (wide segments, b >= 64): __nv_bfloat16 input,
// 8-bit codes in split planes.
#include "rq_launch.cuh"

namespace clq {

cudaError_t launch_rotate_quant_wide_bf16_split(const RotateQuantArgs& a, int logb, int stage,
                                               int threads, size_t smem, int sms,
                                               cudaStream_t st) {
  return rq::launch_rotate_quant_wide_t<__nv_bfloat16, 2>(a, logb, stage, threads, smem, sms, st);
}

}  // namespace clq
