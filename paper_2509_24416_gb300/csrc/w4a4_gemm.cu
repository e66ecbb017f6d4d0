// Launch of the standalone GEMM kernel (gemm_kernel.cuh, instantiated per operand
// family and output type in gemm_*.cu), the weight expansion kernel,
// TMA descriptor helpers and the bounded-wait self test.
#include "gemm_launch.h"
#include "gemm_pipeline.cuh"

#include <cudaTypedefs.h>

#include <atomic>
#include <map>
#include <mutex>
#include <set>
#include <tuple>

namespace clq {

using namespace gemm;

namespace {

// Packed INT4 weights -> E4M3 execution layout (one code per byte, the byte
// is the E4M3 encoding of the integer code).  16 packed bytes per thread.
__global__ void expand_weights_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst,
                                      size_t n16) {
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n16;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const uint4 p = src[i];
    const uint2 e0 = nibbles_to_e4m3(p.x), e1 = nibbles_to_e4m3(p.y);
    const uint2 e2 = nibbles_to_e4m3(p.z), e3 = nibbles_to_e4m3(p.w);
    dst[2 * i] = make_uint4(e0.x, e0.y, e1.x, e1.y);
    dst[2 * i + 1] = make_uint4(e2.x, e2.y, e3.x, e3.y);
  }
}

// Value of an E4M3 byte that holds an integer code (exact): sign, exponent
// with bias 7, three mantissa bits.
__device__ __forceinline__ int e4m3_int(uint32_t byte) {
  const int e = (byte >> 3) & 0xF;
  const int m = byte & 0x7;
  const float v = e == 0 ? 0.f : ldexpf(static_cast<float>(8 + m), e - 10);
  const int i = static_cast<int>(v);
  return (byte & 0x80u) ? -i : i;
}

// Value of the 6-bit E2M3 field f (sign bit 5, exponent bits 4-3 with bias 1,
// three mantissa bits) times 8, exact: an integer code q gives 8 q.
__device__ __forceinline__ int e2m3_times8(uint32_t f) {
  const int e = (f >> 3) & 0x3;
  const int m = f & 0x7;
  const int v = e == 0 ? m : (8 + m) << (e - 1);
  return (f & 0x20u) ? -v : v;
}

// The 16 codes of group g (codes 16 g .. 16 g + 15) of a row in a 4-bit layout
// (packed nibbles, E4M3 bytes or E2M3 fields), as integers; false if a field
// holds no integer (only E2M3 and E4M3 fields can).
__device__ __forceinline__ bool decode_group(const uint8_t* __restrict__ row, int codes, int g,
                                             int (&c)[16]) {
  bool ok = true;
  if (codes == CLQ_CODES_INT4_PACKED) {
    const uint8_t* p = row + 8 * g;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int lo = p[j] & 0xF, hi = p[j] >> 4;
      c[2 * j] = lo >= 8 ? lo - 16 : lo;
      c[2 * j + 1] = hi >= 8 ? hi - 16 : hi;
    }
  } else if (codes == CLQ_CODES_E2M3) {
    const uint8_t* p = row + 12 * g;
    uint64_t lo = 0, hi = 0;  // the 96-bit group, little-endian
#pragma unroll
    for (int j = 0; j < 8; ++j) lo |= static_cast<uint64_t>(p[j]) << (8 * j);
#pragma unroll
    for (int j = 0; j < 4; ++j) hi |= static_cast<uint64_t>(p[8 + j]) << (8 * j);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int bit = 6 * i;
      const uint32_t f = static_cast<uint32_t>(
          (bit < 64 ? (lo >> bit) | (bit > 58 ? hi << (64 - bit) : 0ull) : hi >> (bit - 64)) &
          0x3Full);
      const int v8 = e2m3_times8(f);
      ok &= (v8 & 7) == 0;
      c[i] = v8 / 8;
    }
  } else {
    const uint8_t* p = row + 16 * g;
#pragma unroll
    for (int j = 0; j < 16; ++j) c[j] = e4m3_int(p[j]);
  }
  return ok;
}

// Bytes of one row of K codes in a layout.
__host__ __device__ __forceinline__ size_t codes_row_bytes(int codes, int K) {
  return codes == CLQ_CODES_INT4_PACKED ? static_cast<size_t>(K) / 2
         : codes == CLQ_CODES_E2M3      ? static_cast<size_t>(K) / 4 * 3
         : codes == CLQ_CODES_E4M3_SPLIT ? 2 * static_cast<size_t>(K)
                                         : static_cast<size_t>(K);
}

// One group of 16 integer codes in [-7, 7] into a 4-bit layout.
__device__ __forceinline__ void encode_group(uint8_t* __restrict__ row, int codes, int g,
                                             const int (&c)[16]) {
  if (codes == CLQ_CODES_INT4_PACKED) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      row[8 * g + j] = static_cast<uint8_t>((c[2 * j] & 0xF) | ((c[2 * j + 1] & 0xF) << 4));
  } else if (codes == CLQ_CODES_E2M3) {
    // E2M3 encodings of 0..7: exponent 0 for 0, else 1..3, mantissa in eighths
    constexpr uint8_t kMag[8] = {0x00, 0x08, 0x10, 0x14, 0x18, 0x1A, 0x1C, 0x1E};
    uint64_t lo = 0, hi = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint64_t f = kMag[c[i] < 0 ? -c[i] : c[i]] | (c[i] < 0 ? 0x20u : 0u);
      const int bit = 6 * i;
      if (bit < 64) {
        lo |= f << bit;
        if (bit + 6 > 64) hi |= f >> (64 - bit);
      } else {
        hi |= f << (bit - 64);
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) row[12 * g + j] = static_cast<uint8_t>(lo >> (8 * j));
#pragma unroll
    for (int j = 0; j < 4; ++j) row[12 * g + 8 + j] = static_cast<uint8_t>(hi >> (8 * j));
  } else {
    // E4M3 encodings of 0..7 (exponent bias 7), sign bit 7
    constexpr uint8_t kMag[8] = {0x00, 0x38, 0x40, 0x44, 0x48, 0x4A, 0x4C, 0x4E};
#pragma unroll
    for (int j = 0; j < 16; ++j)
      row[16 * g + j] = kMag[c[j] < 0 ? -c[j] : c[j]] | (c[j] < 0 ? 0x80u : 0u);
  }
}

// Eight E4M3 bytes of integer codes -> packed nibbles.  The magnitudes 0x00 0x38
// 0x40 0x44 0x48 0x4A 0x4C 0x4E of 0 .. 7 differ in the three bits b3 ^ b5, b2 ^ b4,
// b1 ^ b6, which index two byte tables, the codes' nibbles and their negatives'.
// Bytes that are no such code give some nibble in [-7, 7].
__device__ __forceinline__ uint32_t e4m3_to_packed(uint32_t x, uint32_t y) {
  const uint32_t P0 = 0x03010200u, P1 = 0x06070405u;  // 0 2 1 3 5 4 7 6
  const uint32_t N0 = 0x0D0F0E00u, N1 = 0x0A090C0Bu;  // their negatives, mod 16
  auto index = [](uint32_t w) {
    return ((w >> 1) ^ ((w >> 3) & 0x06060606u) ^ ((w >> 6) & 0x01010101u)) & 0x07070707u;
  };
  const uint32_t sel = index(x) | (index(y) << 4);  // nibbles x0 y0 x1 y1 x2 y2 x3 y3
  const uint32_t m0 = prmt(x, y, 0xD9C8u), m1 = prmt(x, y, 0xFBEAu);  // their signs
  const uint32_t lo = (prmt(P0, P1, sel) & ~m0) | (prmt(N0, N1, sel) & m0);
  const uint32_t hi = (prmt(P0, P1, sel >> 16) & ~m1) | (prmt(N0, N1, sel >> 16) & m1);
  // x0 | x1 << 4 and y0 | y1 << 4 in the low bytes of the first, x2.. and y2.. of the other
  return prmt(lo | (lo >> 12), hi | (hi >> 12), 0x5140u);
}

// Code array in one 4-bit layout -> another, one thread a group of 16 codes.
// A code outside [-7, 7] (packed -8) or a field that holds no integer is
// written as 0 and reported.  Between E4M3 bytes and packed nibbles whole words
// are converted, checked by the way back, and only a group that holds something
// else goes code by code; with one byte a load and store the kernel took 24 us for
// 9216 x 3072 codes E4M3 -> packed, 46 back (copying them 6); by whole words with
// arithmetic on the magnitudes 15.4; now 11.4 and 7.3.
__global__ void convert_codes_kernel(const uint8_t* __restrict__ src, int src_codes,
                                     uint8_t* __restrict__ dst, int dst_codes, int rows, int K,
                                     int32_t* status) {
  const int groups = K / 16;
  const size_t n = static_cast<size_t>(rows) * groups;
  const size_t sb = codes_row_bytes(src_codes, K), db = codes_row_bytes(dst_codes, K);
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    if (src_codes == CLQ_CODES_E4M3 && dst_codes == CLQ_CODES_INT4_PACKED) {
      const uint4 w = reinterpret_cast<const uint4*>(src)[i];  // rows are whole groups
      const uint2 o = make_uint2(e4m3_to_packed(w.x, w.y), e4m3_to_packed(w.z, w.w));
      const uint2 a = nibbles_to_e4m3(o.x), b = nibbles_to_e4m3(o.y);
      // magnitudes only: a code's sign went through, and a zero code may carry one
      if ((((w.x ^ a.x) | (w.y ^ a.y) | (w.z ^ b.x) | (w.w ^ b.y)) & 0x7F7F7F7Fu) == 0) {
        reinterpret_cast<uint2*>(dst)[i] = o;
        continue;
      }
    } else if (src_codes == CLQ_CODES_INT4_PACKED && dst_codes == CLQ_CODES_E4M3) {
      const uint2 w = reinterpret_cast<const uint2*>(src)[i];
      // a nibble of 8 (the code -8): its low three bits are zero and its top bit set
      auto minus8 = [](uint32_t x) {
        const uint32_t low = x & 0x77777777u;
        return (~(low + 0x77777777u) & ~low & x & 0x88888888u) != 0;
      };
      if (!(minus8(w.x) || minus8(w.y))) {
        const uint2 a = nibbles_to_e4m3(w.x), b = nibbles_to_e4m3(w.y);
        reinterpret_cast<uint4*>(dst)[i] = make_uint4(a.x, a.y, b.x, b.y);
        continue;
      }
    }
    const size_t r = i / groups;
    const int g = static_cast<int>(i - r * groups);
    int c[16];
    bool ok = decode_group(src + r * sb, src_codes, g, c);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const bool in = c[j] >= -7 && c[j] <= 7;
      ok &= in;
      if (!in) c[j] = 0;
    }
    if (!ok) record_status(status, CLQ_ERR_DEVICE_CODE);
    encode_group(dst + r * db, dst_codes, g, c);
  }
}

// sum_k q[n][k] of each row of a code array (any layout), one warp a row.
__global__ void code_sums_kernel(const uint8_t* __restrict__ W, int codes, int N, int K,
                                 float* __restrict__ wsum) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= N) return;
  if (codes == CLQ_CODES_E2M3) {
    const uint8_t* row = W + static_cast<size_t>(warp) * codes_row_bytes(codes, K);
    int acc = 0;
    for (int gi = lane; gi < K / 16; gi += 32) {
      int c[16];
      decode_group(row, codes, gi, c);
#pragma unroll
      for (int j = 0; j < 16; ++j) acc += c[j];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) wsum[warp] = static_cast<float>(acc);
    return;
  }
  const int width = codes == CLQ_CODES_INT4_PACKED ? K / 2
                    : codes == CLQ_CODES_E4M3_SPLIT ? 2 * K : K;
  const uint4* row = reinterpret_cast<const uint4*>(W + static_cast<size_t>(warp) * width);
  int acc = 0;
  for (int i = lane; i < width / 16; i += 32) {
    const uint4 p = __ldg(row + i);
    const uint32_t w[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t byte = (w[j] >> (8 * k)) & 0xFFu;
        if (codes == CLQ_CODES_INT4_PACKED) {
          const int lo = static_cast<int>(byte & 0xFu), hi = static_cast<int>(byte >> 4);
          acc += (lo >= 8 ? lo - 16 : lo) + (hi >= 8 ? hi - 16 : hi);
        } else {
          acc += e4m3_int(byte);
        }
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) wsum[warp] = static_cast<float>(acc);
}

}  // namespace

cudaError_t launch_code_sums(const uint8_t* W, int codes, int N, int K, float* wsum,
                             cudaStream_t st) {
  const int blocks = (N + 7) / 8;
  code_sums_kernel<<<blocks, 256, 0, st>>>(W, codes, N, K, wsum);
  return cudaGetLastError();
}

bool encode_tma_2d_strided(CUtensorMap* map, CUtensorMapDataType dt, uint32_t esize,
                           const void* base, uint64_t inner, uint64_t rows,
                           uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_rows,
                           CUtensorMapSwizzle swz) {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || p == nullptr)
      return false;
    fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  const cuuint64_t dims[2] = {inner, rows};
  const cuuint64_t strides[1] = {row_stride_bytes};
  const cuuint32_t box[2] = {box_inner, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool encode_tma_2d(CUtensorMap* map, CUtensorMapDataType dt, uint32_t esize, const void* base,
                   uint64_t inner, uint64_t rows, uint32_t box_inner, uint32_t box_rows,
                   CUtensorMapSwizzle swz) {
  return encode_tma_2d_strided(map, dt, esize, base, inner, rows, inner * esize, box_inner,
                               box_rows, swz);
}


bool encode_tma_2d_u8(CUtensorMap* map, const void* base, uint64_t inner_bytes, uint64_t rows,
                      uint32_t box_inner, uint32_t box_rows) {
  return encode_tma_2d(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, base, inner_bytes, rows, box_inner,
                       box_rows, CU_TENSOR_MAP_SWIZZLE_NONE);
}

bool encode_tma_out_tile(CUtensorMap* map, void* Y, int M, int N) {
  return encode_tma_2d(map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Y, static_cast<uint64_t>(N),
                       static_cast<uint64_t>(M), EPI_COLS, EPI_ROWS, CU_TENSOR_MAP_SWIZZLE_64B);
}

int sm_count() {
  static std::atomic<int> cached[64];
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  sms = cached[dev].load(std::memory_order_relaxed);
  if (sms > 0) return sms;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  cached[dev].store(sms, std::memory_order_relaxed);
  return sms;
}

cudaError_t kernel_setup(const void* func, size_t smem, int threads, int* per_sm) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int, size_t, int>, int> occupancy;
  static std::set<std::pair<const void*, int>> raised;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  if (raised.count({func, dev}) == 0) {
    int optin = 0;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, func);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - static_cast<int>(fa.sharedSizeBytes));
    if (e != cudaSuccess) return e;
    raised.insert({func, dev});
  }
  if (per_sm != nullptr) {
    const auto key = std::make_tuple(func, dev, smem, threads);
    auto it = occupancy.find(key);
    if (it == occupancy.end()) {
      int n = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, func, threads, smem);
      if (e != cudaSuccess) return e;
      it = occupancy.emplace(key, n).first;
    }
    *per_sm = it->second;
  }
  return cudaSuccess;
}

// TMA map of a code array (rows x K codes) in any layout: packed boxes of 64
// bytes x box_rows (no swizzle, staged for unpacking), E4M3 boxes of 128
// bytes x box_rows with the 128-byte swizzle (MMA operand), or E2M3 boxes of
// 128 codes x box_rows (96 bytes a row in global memory, 128 in shared
// memory, 128-byte swizzle; K a multiple of 128).  For the split
// layout ([rows][2][K]) the map covers plane `plane` of every row (row stride
// 2K bytes); for the others `plane` must be 0.
bool encode_codes_map(CUtensorMap* map, const uint8_t* base, int codes, int rows, int K,
                      int box_rows, int plane) {
  if (codes == CLQ_CODES_E2M3)  // 16 codes in 12 bytes, each group padded to 16 in smem
    return encode_tma_2d_strided(map, CU_TENSOR_MAP_DATA_TYPE_16U6_ALIGN16B, 1, base,
                                 static_cast<uint64_t>(K), static_cast<uint64_t>(rows),
                                 static_cast<uint64_t>(K) / 4 * 3, BK, box_rows,
                                 CU_TENSOR_MAP_SWIZZLE_128B);
  if (codes == CLQ_CODES_INT4_PACKED)
    return encode_tma_2d_u8(map, base, static_cast<uint64_t>(K) / 2, static_cast<uint64_t>(rows),
                            BKP, box_rows);
  const bool split = codes == CLQ_CODES_E4M3_SPLIT;
  return encode_tma_2d_strided(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1,
                               base + (split ? static_cast<size_t>(plane) * K : 0),
                               static_cast<uint64_t>(K), static_cast<uint64_t>(rows),
                               static_cast<uint64_t>(K) * (split ? 2 : 1), BK, box_rows,
                               CU_TENSOR_MAP_SWIZZLE_128B);
}

namespace {

// Clocks a K step of a pair's tile of bn columns takes with 1, 2 or 4 products of
// code planes (a single CTA: 740 and 1200 at 256 columns, 1300 at 128 with four),
// fitted to 434 measured products.
double pair_step(int products, int bn) {
  if (products == 4) return bn == 64 ? 766 : 1146;
  if (products == 2) return bn == 64 ? 520 : bn == 128 ? 630 : 1128;
  return bn == 64 ? 300 : bn == 128 ? 390 : bn == 192 ? 458 : 587;
}

// Clocks of a product by the model of gemm_tile_n.
double tiles_cost(int M, int N, int K, int rows, int units, int bn, double step, int epi) {
  const long tiles = static_cast<long>((M + rows - 1) / rows) * ((N + bn - 1) / bn);
  const long rounds = (tiles + units - 1) / units;
  const double drain = epi * bn / 64.0;
  return rounds * std::max((K + BK - 1) / BK * step, drain + 500) + drain;
}

}  // namespace

// Tile width of execution-layout operands, `units` CTAs or CTA pairs walking tiles
// of `rows` rows.  The units go ceil(tiles / units) rounds; a tile takes its K
// steps (clocks a step of a pair's main loop, measured alone: 587 / 458 / 390 for
// 256 / 192 / 128 columns, and what 20 KB of operands take to arrive for 64) or
// its epilogue, whichever is longer, and the last one's epilogue comes on top
// (`epi` clocks for each 64 columns: 1000 with eight epilogue warps, 1100 with the
// fused kernel's four).  256 wins on large products, 192 where N splits into its
// tiles with no more rounds (N = 1152: 6 x 192 instead of 4.5 x 256), 128 and 64
// where the wider tiles leave units idle (us at 256 / 192 / 128 / 64 columns: 256 x
// 1152 x 1152 6.8 / 5.8 / 4.9 / 4.4, 256 x 3072 x 12288 29.6 / 22.9 / 16.4 / 16.1,
// 1024 x 4608 x 1152 7.8 / 8.1 / 7.6 / 9.6, 2048 x 4608 x 1152 10.6 / 10.6 / 11.0 /
// 15.1, 8192 x 1152 x 4608 34.0 / 27.6 / 28.0 / 44.6; this rule is within 4 % of
// the best of them on 15 such shapes in each layout).  `narrow`: 64 and 128 are
// built for these operands; `mid`: 192 is.
int gemm_tile_n(int M, int N, int K, int rows, int units, bool mid, bool narrow, int epi) {
  const int width[4] = {256, 192, 128, 64};
  int best = BN;
  double best_cost = 1e300;
  for (int i = 0; i < 4; ++i) {
    if ((width[i] == 192 && !mid) || (width[i] < 192 && !narrow)) continue;
    const double cost = tiles_cost(M, N, K, rows, units, width[i], pair_step(1, width[i]), epi);
    if (cost < best_cost) {
      best_cost = cost;
      best = width[i];
    }
  }
  return best;
}

// Whether the widest tile of a single CTA beats the pairs' tile of `pair_bn` columns;
// `products`: products of code planes a K step (1, 2 for W4A8, 4 for W8A8).  Pairs win
// large products, but with twice the rows a tile their rounds come out coarser: 3129
// rows x 12288 -> 3072, W4A8, takes three rounds of 256 x 256 (161 us) or two of 128 x
// 256 (123); 375 x 5376 -> 4960, W8A8, 50.5 us or 30.0; 300 x 3072 -> 12288 14.8 or
// 12.4, W4A8 24.7 or 17.7.  And activation codes of less than 128 KB starve pairs more
// than single CTAs (3072 -> 12288: 12.6 us with 16 to 32 rows, 9.7 with 48; as single
// CTAs 11.5 to 11.9 and 11.4), by about 10 clocks a step for each pair that reads
// them: 4 x 896 -> 11479, W4A8, 14.0 or 9.1; 1 x 8512 -> 10112 36.7 or 26.1
// (`few_starve`; not in the fused kernel: 2 x 10816 -> 11616 47.7, single 62.5).  The
// margin of 10 % covers what the model leaves open: of 678 products of 1 .. 16384
// rows, at random, the rule moves 26, all of them to a tile at least as fast.
bool single_cta_wins(int M, int N, int K, int products, int pair_bn, int sms, bool few_starve) {
  const double codes = static_cast<double>(M) * K * (products == 1 ? 1 : 2);
  const int readers = std::min((N + pair_bn - 1) / pair_bn, sms / 2);
  const double starved = few_starve && codes < 131072 ? 10.0 * readers : 0.0;
  const int epi = 1000;
  const double pair = tiles_cost(M, N, K, 2 * BM, sms / 2, pair_bn,
                                 pair_step(products, pair_bn) + starved, epi);
  const double one =
      products == 4 ? tiles_cost(M, N, K, BM, sms, 128, 1300, epi)
                    : tiles_cost(M, N, K, BM, sms, BN, products == 2 ? 1200 : 740, epi);
  return 1.1 * one < pair;
}

cudaError_t launch_w4a4_gemm(const uint8_t* Xq, int x_codes, const uint8_t* W, int w_codes,
                             const GemmArgs& g, int out_dtype, cudaStream_t st) {
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  const bool apack = x_codes == CLQ_CODES_INT4_PACKED;
  const bool bpack = w_codes == CLQ_CODES_INT4_PACKED;
  const bool split = x_codes == CLQ_CODES_E4M3_SPLIT || w_codes == CLQ_CODES_E4M3_SPLIT;
  const bool w8a8 = x_codes == CLQ_CODES_E4M3_SPLIT && w_codes == CLQ_CODES_E4M3_SPLIT;
  // Operands in an execution layout run on CTA pairs (tcgen05 cta_group::2) unless
  // single_cta_wins: each CTA loads its 128 rows of A and half of B's rows, so a K step brings 32 KB
  // into an SM instead of 48, six stages fit instead of four, and the L2 reads
  // and power of a product fall with them (measured against single CTAs with
  // the same epilogue: 8192 x 3456 x 1152 26.8 -> 23.5 us, 4608 x 3072 x 12288
  // 110.5 -> 84.6, 65536 x 12288 x 3072 1523 -> 1235; 20 x 480 x 1920 6.9 -> 6.4).
  TileShape t{apack || bpack ? 1 : 2, BN};
  if (w8a8) {
    // 128 columns (two or three accumulators of them fill tensor memory), 64 where
    // that leaves pairs idle and the product's accumulators allow it
    t.bn = 128;
    const int pairs = ((g.M + t.cg * BM - 1) / (t.cg * BM)) * ((g.N + 127) / 128);
    if (g.lo == nullptr && g.K <= kSep2MaxK && 2 * pairs <= sms / t.cg) t.bn = 64;
  }
  else if (!apack && !bpack && !(split && g.lo != nullptr))
    t.bn = gemm_tile_n(g.M, g.N, g.K, t.cg * BM, sms / t.cg, !split && g.lo == nullptr, true);
  if (t.cg == 2 && single_cta_wins(g.M, g.N, g.K, w8a8 ? 4 : split ? 2 : 1, t.bn, sms))
    t = {1, w8a8 ? 128 : BN};
  MapSet m;
  const int brows = t.bn / t.cg;  // each CTA of a pair loads half of B
  if (!encode_codes_map(&m.A, Xq, x_codes, g.M, g.K, BM, 0) ||
      !encode_codes_map(&m.B, W, w_codes, g.N, g.K, brows, 0))
    return cudaErrorInvalidValue;
  m.A2 = m.A;  // unused unless split
  m.B2 = m.B;
  if (x_codes == CLQ_CODES_E4M3_SPLIT && !encode_codes_map(&m.A2, Xq, x_codes, g.M, g.K, BM, 1))
    return cudaErrorInvalidValue;
  if (w_codes == CLQ_CODES_E4M3_SPLIT && !encode_codes_map(&m.B2, W, w_codes, g.N, g.K, brows, 1))
    return cudaErrorInvalidValue;
  const int use_tma_store = (g.N % 8 == 0) ? 1 : 0;
  if (use_tma_store) {
    if (!encode_tma_out_tile(&m.Y, g.Y, g.M, g.N)) return cudaErrorInvalidValue;
  } else {
    m.Y = m.A;  // unused
  }
  const int tiles = ((g.M + t.cg * BM - 1) / (t.cg * BM)) * ((g.N + t.bn - 1) / t.bn);
  const int grid = t.cg * std::min(tiles, sms / t.cg);
  const bool f16 = out_dtype == CLQ_F16;
  auto* go = apack || bpack                ? (f16 ? launch_gemm_packed_f16 : launch_gemm_packed_bf16)
             : x_codes == CLQ_CODES_E2M3   ? (f16 ? launch_gemm_e2m3_f16 : launch_gemm_e2m3_bf16)
             : split || g.lo != nullptr    ? (f16 ? launch_gemm_bits_f16 : launch_gemm_bits_bf16)
                                           : (f16 ? launch_gemm_e4m3_f16 : launch_gemm_e4m3_bf16);
  return go(m, g, x_codes, w_codes, t, use_tma_store, grid, st);
}

cudaError_t launch_convert_codes(const uint8_t* src, int src_codes, uint8_t* dst, int dst_codes,
                                 int rows, int K, int32_t* status, cudaStream_t st) {
  const size_t n = static_cast<size_t>(rows) * (K / 16);
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  const int blocks = static_cast<int>(std::min<size_t>((n + 255) / 256, 8u * sms));
  convert_codes_kernel<<<std::max(blocks, 1), 256, 0, st>>>(src, src_codes, dst, dst_codes, rows,
                                                            K, status);
  return cudaGetLastError();
}

cudaError_t launch_expand_weights(const uint8_t* Wq, int N, int K, uint8_t* We, cudaStream_t st) {
  const size_t n16 = static_cast<size_t>(N) * (K / 2) / 16;
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  const int blocks = static_cast<int>(std::min<size_t>((n16 + 255) / 256, 8u * sms));
  expand_weights_kernel<<<std::max(blocks, 1), 256, 0, st>>>(
      reinterpret_cast<const uint4*>(Wq), reinterpret_cast<uint4*>(We), n16);
  return cudaGetLastError();
}

// ------------------------------------------------------ bounded-wait test ---
namespace {
__global__ void wait_selftest_kernel(uint64_t timeout_ns, int32_t* status) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int32_t abort;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort = 0;
    fence_mbarrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait_bounded(&bar, 0, &abort, status, timeout_ns);
  __syncthreads();
}
}  // namespace

cudaError_t launch_wait_selftest(uint64_t timeout_ns, int32_t* status, cudaStream_t st) {
  wait_selftest_kernel<<<1, 32, 0, st>>>(timeout_ns, status);
  return cudaGetLastError();
}

}  // namespace clq
