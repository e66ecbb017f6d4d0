// Outlier scores under the alternative metrics of arxiv 2509.24416 Sec. 4.4
// ("Choice of Outlier Metric": percentile (1 %, 99 %), top-k mean with
// k = 1 %, range, peak-to-average ratio), next to Sec. 3.3's absolute
// maximum.  Offline, once per layer.  The scores decide an integer
// permutation, so every step is taken in fp32 in one fixed order, the one
// the CPU oracle takes:
//   S[t] = (sum over b in order of calib[b][t][c]) / B;
//   absmax     max_t |S|;
//   range      max_t S - min_t S;
//   par        max_t |S| / ((sum over t in order of |S|) / T), 0 if the sum is 0;
//   percentile max(|P(0.01)|, |P(0.99)|), P(q) = v[lo] + (pos - lo)(v[lo+1] - v[lo])
//              over the ascending order statistics v, pos = q (T - 1), lo = floor(pos);
//   topk_mean  (sum of the k largest |S|, largest first) / k, k = max(1, (T + 50) / 100).
// One CTA per channel holds S (T <= 16384 values) in shared memory and sorts
// it with a bitonic network where an order statistic is needed.
#include "clq_device.cuh"
#include "clq_kernels.h"
#include "sort_util.cuh"

namespace clq {

namespace {

constexpr int kThreads = 256;

// Block-wide max of x (every thread contributes); the result in every thread.
__device__ __forceinline__ float block_max(float x, float* red) {
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) red[w] = x;
  __syncthreads();
  float r = red[0];
  for (int i = 1; i < kThreads / 32; ++i) r = fmaxf(r, red[i]);
  __syncthreads();
  return r;
}

__device__ __forceinline__ float percentile_fp32(const float* v, int n, float q) {
  const float pos = __fmul_rn(q, static_cast<float>(n - 1));
  const int lo = static_cast<int>(floorf(pos));
  const int hi = min(lo + 1, n - 1);
  const float frac = __fsub_rn(pos, static_cast<float>(lo));
  return __fadd_rn(v[lo], __fmul_rn(frac, __fsub_rn(v[hi], v[lo])));
}

template <typename T>
__global__ void __launch_bounds__(kThreads) outlier_metric_kernel(const uint16_t* calib, int B,
                                                                  int Tn, int K, int Tp,
                                                                  int metric, float* scores) {
  extern __shared__ float v[];  // [Tp]
  __shared__ float red[kThreads / 32];
  const int c = blockIdx.x;
  const size_t bstride = static_cast<size_t>(Tn) * K;
  const float fb = static_cast<float>(B);
  // S[t], and what the metric sorts: S (percentile), -|S| (top-k: ascending
  // order puts the largest magnitudes first).  Padding sorts to the end.
  float lmax = 0.f, lmin = 0.f, labs = 0.f;
  bool any = false;
  for (int t = threadIdx.x; t < Tp; t += blockDim.x) {
    float x = 0.f;
    if (t < Tn) {
      float s = 0.f;
      for (int b = 0; b < B; ++b)
        s = __fadd_rn(s, Num<T>::to_f(calib[b * bstride + static_cast<size_t>(t) * K + c]));
      x = __fdiv_rn(s, fb);
      lmax = any ? fmaxf(lmax, x) : x;
      lmin = any ? fminf(lmin, x) : x;
      labs = fmaxf(labs, fabsf(x));
      any = true;
    }
    if (metric == CLQ_METRIC_TOPK_MEAN)
      v[t] = t < Tn ? -fabsf(x) : __int_as_float(0x7f800000);  // +inf pad
    else
      v[t] = t < Tn ? x : __int_as_float(0x7f800000);
  }
  __syncthreads();
  // Block extremes (threads without a token hold neutral values).
  const float mx = block_max(any ? lmax : -__int_as_float(0x7f800000), red);
  const float mn = -block_max(any ? -lmin : -__int_as_float(0x7f800000), red);
  const float peak = block_max(labs, red);
  if (metric == CLQ_METRIC_PERCENTILE || metric == CLQ_METRIC_TOPK_MEAN)
    bitonic_sort_ascending(v, Tp);
  if (threadIdx.x != 0) return;
  float out = 0.f;
  switch (metric) {
    case CLQ_METRIC_ABSMAX:
      out = peak;
      break;
    case CLQ_METRIC_RANGE:
      out = __fsub_rn(mx, mn);
      break;
    case CLQ_METRIC_PAR: {
      float sum = 0.f;
      for (int t = 0; t < Tn; ++t) sum = __fadd_rn(sum, fabsf(v[t]));
      const float mean = __fdiv_rn(sum, static_cast<float>(Tn));
      out = mean > 0.f ? __fdiv_rn(peak, mean) : 0.f;
      break;
    }
    case CLQ_METRIC_PERCENTILE: {
      const float lo = percentile_fp32(v, Tn, 0.01f);
      const float hi = percentile_fp32(v, Tn, 0.99f);
      out = fmaxf(fabsf(lo), fabsf(hi));
      break;
    }
    default: {  // CLQ_METRIC_TOPK_MEAN
      const int k = max(1, (Tn + 50) / 100);
      float sum = 0.f;
      for (int i = 0; i < k; ++i) sum = __fadd_rn(sum, -v[i]);
      out = __fdiv_rn(sum, static_cast<float>(k));
      break;
    }
  }
  scores[c] = out;
}

}  // namespace

cudaError_t launch_outlier_metric(const void* calib, int dtype, int B, int T, int K, int metric,
                                  float* scores, cudaStream_t st) {
  int Tp = 1;
  while (Tp < T) Tp <<= 1;
  const size_t smem = static_cast<size_t>(Tp) * sizeof(float);
  const uint16_t* c = static_cast<const uint16_t*>(calib);
  if (dtype == CLQ_F16) {
    auto k = outlier_metric_kernel<__half>;
    cudaError_t e = kernel_setup(reinterpret_cast<const void*>(k), smem, kThreads, nullptr);
    if (e != cudaSuccess) return e;
    k<<<K, kThreads, smem, st>>>(c, B, T, K, Tp, metric, scores);
  } else {
    auto k = outlier_metric_kernel<__nv_bfloat16>;
    cudaError_t e = kernel_setup(reinterpret_cast<const void*>(k), smem, kThreads, nullptr);
    if (e != cudaSuccess) return e;
    k<<<K, kThreads, smem, st>>>(c, B, T, K, Tp, metric, scores);
  }
  return cudaGetLastError();
}

namespace {

constexpr int kPermThreads = 1024;
constexpr int kPermPer = 16;  // channels a thread, K <= 16384

// Sums of (x, y) over the block, in every thread, through red (32 entries that
// nothing else reads or writes until the next barrier but one).
__device__ __forceinline__ int2 block_sum2(int x, int y, int2* red) {
  x = __reduce_add_sync(0xffffffffu, x);
  y = __reduce_add_sync(0xffffffffu, y);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[w] = make_int2(x, y);
  __syncthreads();
  const int2 r = red[lane];
  return make_int2(__reduce_add_sync(0xffffffffu, r.x), __reduce_add_sync(0xffffffffu, r.y));
}

// The column-swap vector (Sec. 3.3, "Outlier Detection") from scores on the
// device: the K / 2 channels of the highest scores, ties to the lower index, in
// ascending order, then the others.  One block: the K / 2-th largest score by a
// search on order-preserving keys, two bits a round (three block-wide counts, two
// of them in one word), until a threshold has just K / 2 keys at or above it; the
// ties and the positions by one prefix sum over the channels, which threads own in
// index order.  It takes the place of a copy to the host, a sort there (157 us for
// K = 3072) and a copy back.  A chain of latencies on one SM: with a bit a round,
// two barriers each, and all sixteen channels of a thread counted it took 17.0 us
// at K = 3072, now 10.6.  NaN scores: *bad = 1 and the identity.
__global__ void __launch_bounds__(kPermThreads) build_permutation_kernel(
    const float* __restrict__ scores, int K, int32_t* __restrict__ perm,
    int32_t* __restrict__ bad) {
  __shared__ int2 red[3][32];  // alternating in the search, the last for the prefix sum
  pdl_launch_dependents();     // the kernel that orders this one's writes
  const int per = (K + kPermThreads - 1) / kPermThreads;
  const int k0 = static_cast<int>(threadIdx.x) * per;
  const int h = K / 2;
  uint32_t key[kPermPer];
  int nan = 0;
#pragma unroll
  for (int i = 0; i < kPermPer; ++i) {
    key[i] = 0;  // below every float's key
    if (i < per && k0 + i < K) {
      const float f = scores[k0 + i] + 0.0f;  // -0 equals 0
      nan |= f != f;
      const uint32_t u = __float_as_uint(f);
      key[i] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    }
  }
  nan = __syncthreads_or(nan);
  if (threadIdx.x == 0) *bad = nan ? 1 : 0;
  // at least h keys are at or above it, at last just h or the h-th largest key
  uint32_t cut = h > 0 ? 0u : ~0u;
  for (int bit = 30; bit >= 0 && h > 0; bit -= 2) {
    const uint32_t one = 1u << bit;
    int c1 = 0, c23 = 0;  // counts up to 16384 in 16 bits
#pragma unroll
    for (int i = 0; i < kPermPer; ++i) {
      if (i >= per) break;
      c1 += key[i] >= (cut | one);
      c23 += (key[i] >= (cut | (2 * one)) ? 1 : 0) + (key[i] >= (cut | (3 * one)) ? 65536 : 0);
    }
    const int2 n = block_sum2(c1, c23, red[(bit >> 1) & 1]);
    const int n1 = n.x, n2 = n.y & 0xFFFF, n3 = n.y >> 16;
    const int j = n3 >= h ? 3 : n2 >= h ? 2 : n1 >= h ? 1 : 0;
    cut |= static_cast<uint32_t>(j) << bit;
    if (j > 0 && (j == 3 ? n3 : j == 2 ? n2 : n1) == h) break;  // no tie to settle
  }
  int mine = 0;  // keys above the cut, and at it times 65536
#pragma unroll
  for (int i = 0; i < kPermPer; ++i) {
    if (i >= per) break;
    mine += (key[i] > cut ? 1 : 0) + (key[i] == cut ? 65536 : 0);
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int sum = mine;  // over the threads of the warp up to this one
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, sum, o);
    if (lane >= o) sum += t;
  }
  if (lane == 31) red[2][w].x = sum;
  __syncthreads();
  const int warp_sum = red[2][lane].x;
  const int before = __reduce_add_sync(0xffffffffu, lane < w ? warp_sum : 0) + sum - mine;
  // of the channels at the cut, the first `left` are high
  const int left = h - (__reduce_add_sync(0xffffffffu, warp_sum) & 0xFFFF);
  int rank = before >> 16;                            // channels at the cut before this one
  int pos = (before & 0xFFFF) + (rank < left ? rank : left);  // high channels before it
#pragma unroll
  for (int i = 0; i < kPermPer; ++i) {
    const int k = k0 + i;
    if (i >= per || k >= K) break;
    const bool at = key[i] == cut;
    const bool hi = key[i] > cut || (at && rank < left);
    if (nan)
      perm[k] = k;
    else
      perm[hi ? pos : h + (k - pos)] = k;
    rank += at;
    pos += hi;
  }
}

// Behind the builder: waits until that has completed and its writes are visible, and
// ends.  Rotate-quant and the fused kernel read the swap vector before their
// programmatic-launch wait; they can start no earlier than this kernel ends, so a
// vector built just before them on the stream is the one they read.  It becomes
// resident while the builder runs: launched plainly it made a calibration of 122 us
// about 5 us longer, this way about 3.
__global__ void order_swap_vector_kernel() { pdl_wait(); }

}  // namespace

cudaError_t launch_build_permutation(const float* scores, int K, int32_t* perm, int32_t* bad,
                                     cudaStream_t st) {
  build_permutation_kernel<<<1, kPermThreads, 0, st>>>(scores, K, perm, bad);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_pdl(order_swap_vector_kernel, 1, 32, 0, st);
}

}  // namespace clq
