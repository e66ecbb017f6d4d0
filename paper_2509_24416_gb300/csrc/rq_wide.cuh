// Wide-segment rotate-quantize: the hot-path variant of the tile loop for
// 4-bit (E4M3, E2M3) and 8-bit (split-plane) codes when b >= 64 (the OBS transform of arxiv 2509.24416
// Sec. 3.3 and the per-token quantization of Sec. 3.1 / Eq. 1, symmetric, or
// asymmetric with the row's minimum and maximum, as in rq_device.cuh).
//
// Each thread owns 64 consecutive permuted positions of one row, so a block
// of b = 64 is transformed entirely in its registers; b = 128 / 256 add one /
// two stages across lanes that exchange half of the registers each.  The
// cross-lane shuffles, which load the shared-memory pipe as much as the gather
// does, so drop out (b = 64), or come to half / one an element instead of two /
// three with 32-wide segments.  The 64 gather offsets (bytes from the stage
// start, below 64 KB) are kept two to a register, so the thread holds as many
// address registers as the 32-wide loop while doing twice the work per tile.  The
// rest follows rq_pair.cuh: round-robin tiles, STAGES stages in flight,
// three-input maxima, one CTA barrier per tile, the XOR-ordered gather whose sign
// flips the store undoes, and a prologue that runs while the previous kernel
// drains: barriers, an L2 prefetch of the first tiles and the gather offsets from
// the swap vector (a layer constant), with X read only after the
// programmatic-launch wait.
//
// What bounds it: the gather (one 16-bit load an element at scattered columns,
// about 3 wavefronts a load) and the latencies that 12 warps a SM leave exposed.
// Measured, back to back, E4M3 codes: 8192 x 1152 8.2 / 9.4 us at b = 64 / 128
// (copies alone 3.5), 65536 x 1152 44.4 / 52.4, 4608 x 12288 37.5 / 42.2; with
// 32-wide segments b = 128 took 11.2, 63.0 and 53.2.
#pragma once

#include "rq_pair.cuh"

namespace clq {
namespace rq {

constexpr int kWideMaxRegs = 168;

// Shared memory of the wide loop: STAGES stages of STAGE bytes, row maxima
// and (asymmetric codes) row minima [3][RH] each, STAGES barriers, abort flag.
__host__ __device__ inline size_t wide_smem_bytes(int RH, int stage, int stages) {
  return static_cast<size_t>(stages) * stage + 24u * RH + 8u + 8u * stages + 16u;
}

// max_k v[k] and min_k v[k] over a thread's 64 values: four chains of three-input
// maxima and minima (a tree's intermediate values cost registers that the loop
// does not have).
__device__ __forceinline__ void wide_minmax(const float2 (&v)[32], float& mx, float& mn) {
  float a[4], b[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    a[i] = fmaxf(v[i].x, v[i].y);
    b[i] = fminf(v[i].x, v[i].y);
  }
#pragma unroll
  for (int i = 4; i < 32; ++i) {
    a[i & 3] = max3(a[i & 3], v[i].x, v[i].y);
    b[i & 3] = min3(b[i & 3], v[i].x, v[i].y);
  }
  mx = fmaxf(max3(a[0], a[1], a[2]), a[3]);
  mn = fminf(min3(b[0], b[1], b[2]), b[3]);
}

// max_k |v[k]| over a thread's 64 values, the same way.
__device__ __forceinline__ float wide_absmax(const float2 (&v)[32]) {
  float m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = fmaxf(fabsf(v[i].x), fabsf(v[i].y));
#pragma unroll
  for (int i = 4; i < 32; ++i) m[i & 3] = max3_abs(m[i & 3], v[i].x, v[i].y);
  return fmaxf(max3(m[0], m[1], m[2]), m[3]);
}

// Butterfly stages of a 64-wide segment: strides 2 .. 32 in registers (v[k]
// holds positions 2k, 2k + 1, stride 1 done), then strides 64 .. b / 2 across the
// 2 or 4 lanes of a block, each stage exchanging half of the registers: lane l
// and its partner l ^ 1 (l ^ 2) each keep the outputs of one half of the index
// range, send the other half and form both the sum and the difference of what
// they then hold, 32 shuffles a stage where keeping one's own segment takes 64.
// For the partner to hold the other half in the same registers, the last
// in-register stages of a lane with that bit set leave their sum and difference
// swapped (a multiplication by -1 that rounds nothing).  Every output is the same
// sum, rounded in the same order, as with whole segments; differences in lanes
// with the bit set come out negated, which wide_flip accounts for.
//
// Where a register ends up: with X = log2(b) - 6 stages across lanes, register
// chunk c (registers 16 c .. 16 c + 15) holds the block's positions
// wide_chunk<X>(c, lane) .. + 15.
template <int LOGB>
__device__ __forceinline__ void wide_butterflies(float2 (&v)[32], int lane) {
  const float2 neg1 = make_float2(-1.f, -1.f);
#pragma unroll
  for (int hp = 1; hp < 8; hp <<= 1)
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if ((k & hp) == 0) {
        const float2 x0 = v[k], x1 = v[k + hp];
        v[k] = __fadd2_rn(x0, x1);
        v[k + hp] = __ffma2_rn(x1, neg1, x0);
      }
#pragma unroll
  for (int hp = 8; hp < 32; hp <<= 1) {
    constexpr int X = LOGB - 6;
    const int bit = hp == 16 ? 1 : 2;  // lane bit that swaps this stage's outputs
    if (X >= (hp == 16 ? 1 : 2)) {
      const float sg = (lane & bit) ? -1.f : 1.f;
      const float2 p = make_float2(sg, sg), m = make_float2(-sg, -sg);
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if ((k & hp) == 0) {
          const float2 x0 = v[k], x1 = v[k + hp];
          v[k] = __ffma2_rn(x1, p, x0);
          v[k + hp] = __ffma2_rn(x1, m, x0);
        }
    } else {
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if ((k & hp) == 0) {
          const float2 x0 = v[k], x1 = v[k + hp];
          v[k] = __fadd2_rn(x0, x1);
          v[k + hp] = __ffma2_rn(x1, neg1, x0);
        }
    }
  }
#pragma unroll
  for (int x = 0; x < LOGB - 6; ++x) {
    const int hp = 16 >> x;  // keep v[k], send v[k + hp]
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if ((k & hp) == 0) {
        float2 q;
        q.x = __shfl_xor_sync(0xffffffffu, v[k + hp].x, 1 << x);
        q.y = __shfl_xor_sync(0xffffffffu, v[k + hp].y, 1 << x);
        const float2 own = v[k];
        v[k] = __fadd2_rn(own, q);
        v[k + hp] = __ffma2_rn(q, neg1, own);
      }
  }
}

// First position, within the block of b = 64 << X, of register chunk c (16
// registers) after wide_butterflies.
template <int X>
__device__ __forceinline__ int wide_chunk(int c, int lane) {
  if (X == 0) return 16 * c;
  if (X == 1) return (c >> 1) * 64 + (lane & 1) * 32 + (c & 1) * 16;
  return (c & 1) * 128 + (c >> 1) * 64 + (lane & 1) * 32 + ((lane >> 1) & 1) * 16;
}

// Bit q: registers 4 q .. 4 q + 3 hold the negated transform, from the XOR order
// xm of the gather (output i of a segment gets the sign (-1)^popc(i & xm)) and
// from the differences of the lanes whose bit is set.
template <int X>
__device__ __forceinline__ uint32_t wide_flip(int xm, int lane) {
  uint32_t flip = 0;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int c = q >> 2;
    const int i = (wide_chunk<X>(c, lane) & 63) + 4 * (q & 3);
    int neg = __popc(i & xm);
    if (X >= 1) neg += (c >> 1) & lane;
    if (X >= 2) neg += c & (lane >> 1);
    flip |= static_cast<uint32_t>(neg & 1) << q;
  }
  return flip;
}

// 1.5 * 2^23 + 8: a code q added to it by an fma comes out rounded (ties to even:
// the constant is even) as q + 8 in the low mantissa bits.
constexpr float kSplitMagic = 12582920.0f;

// Split-plane stores of a thread's 64 codes, v holding q + kSplitMagic (SCALE:
// values that +-rcp, by the bits of flip, turns into it): 16 h = floor((q + 8) /
// 16) * 16 by one addition that rounds down at 16, the ulp of 1.5 * 2^27, then l =
// q - 16 h, both exact; E4M3 bytes, 16 codes a store and plane.
template <int X, bool SCALE>
__device__ __forceinline__ void wide_store_split(const RotateQuantArgs& a, float2 (&v)[32],
                                                 int row, int block, int lane, float rcp,
                                                 uint32_t flip) {
  const int K = a.K;
  constexpr float big = 201326592.0f;  // 1.5 * 2^27
  constexpr float up = big - 12582912.0f;
  uint8_t* qrow = a.Q + static_cast<size_t>(row) * 2 * K + block;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t wh[4], wl[4];
    // one chunk after the other: interleaved, their temporaries spill
    asm volatile("" : "+r"(flip)::"memory");
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint16_t eh[2], el[2];
      const float rs = ((flip >> (4 * c + j)) & 1u) ? -rcp : rcp;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        float2 x = v[8 * c + 2 * j + i];
        if (SCALE)
          x = __ffma2_rn(x, make_float2(rs, rs), make_float2(kSplitMagic, kSplitMagic));
        const float2 h16 = __fadd2_rn(__fadd2_rd(x, make_float2(up, up)), make_float2(-big, -big));
        const float2 q = __fadd2_rn(x, make_float2(-kSplitMagic, -kSplitMagic));
        const float2 l = __ffma2_rn(h16, make_float2(-1.f, -1.f), q);
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(eh[i]) : "f"(h16.y), "f"(h16.x));
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(el[i]) : "f"(l.y), "f"(l.x));
      }
      wh[j] = static_cast<uint32_t>(eh[0]) | (static_cast<uint32_t>(eh[1]) << 16);
      wl[j] = static_cast<uint32_t>(el[0]) | (static_cast<uint32_t>(el[1]) << 16);
    }
    uint8_t* q = qrow + wide_chunk<X>(c, lane);
    *reinterpret_cast<uint4*>(q) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
    *reinterpret_cast<uint4*>(q + K) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
  }
}

// The same for a row with a subnormal scale s: exact divisions, as in rq_device.cuh.
// A call of its own, on a copy of the values: as a branch of the hot path it cost
// that path 80 bytes of spills.
template <int X>
static __device__ __noinline__ void wide_store_split_tiny(uint8_t* qrow, int K, const float2* t,
                                                          float s, uint32_t flip, int lane) {
#pragma unroll 1
  for (int r = 0; r < 64; ++r) {
    const float v = __fdiv_rn((r & 1) ? t[r >> 1].y : t[r >> 1].x, s);
    const float x = (((flip >> (r >> 2)) & 1u) ? -v : v) + kSplitMagic;
    const float q = x - kSplitMagic;
    const float h16 = 16.f * floorf((q + 8.f) * 0.0625f);
    uint16_t eh, el;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(eh) : "f"(0.f), "f"(h16));
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(el) : "f"(0.f), "f"(q - h16));
    uint8_t* at = qrow + wide_chunk<X>(r >> 4, lane) + (r & 15);
    at[0] = static_cast<uint8_t>(eh);
    at[K] = static_cast<uint8_t>(el);
  }
}

// Scale, codes and stores of one row's 64 values of a thread; `am` is the row's
// |x| maximum; bit q of `flip` flips the signs of registers 4q .. 4q + 3.
template <int CODES, bool ROT, int X>
__device__ __forceinline__ void wide_quant_store(const RotateQuantArgs& a, float2 (&v)[32],
                                                 int row, int seg, float am, uint32_t flip,
                                                 int lane) {
  const int K = a.K;
  const int block = (seg >> X) << (6 + X);  // first position of the thread's block
  // s = am / qmax by division by a constant known in advance (Brisebarre,
  // Muller and Raina, IEEE Trans. Computers 53(8), 2004), as in rq_device.cuh
  constexpr float qmax = CODES == 2 ? 127.0f : 7.0f;
  constexpr float rdiv = 1.0f / qmax;
  const float q1 = am * rdiv;
  const float s_row = fmaf(fmaf(-qmax, q1, am), rdiv, q1);
  if (seg == 0) a.S[row] = s_row;
  if (ROT) {
    float* dst = a.rot + static_cast<size_t>(row) * K + block;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const float sg = ((flip >> q) & 1u) ? -1.f : 1.f;
      *reinterpret_cast<float4*>(dst + wide_chunk<X>(q >> 2, lane) + 4 * (q & 3)) =
          make_float4(sg * v[2 * q].x, sg * v[2 * q].y, sg * v[2 * q + 1].x, sg * v[2 * q + 1].y);
    }
  }
  // v <- rint(v / s) + 1.5 * 2^23 (ties to even), v / s as v * rcp(s); a zero
  // row gets zero codes; a subnormal s takes exact divisions with 8-bit codes, and
  // is scaled with v by 2^64 first with 4-bit ones.
  if constexpr (CODES == 2) {
    if (s_row > 0.f && s_row < 1.17549435e-38f) {
      float2 t[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) t[k] = v[k];
      wide_store_split_tiny<X>(a.Q + static_cast<size_t>(row) * 2 * K + block, K, t, s_row, flip,
                               lane);
      return;
    }
    const float rcp = s_row > 0.f ? rcp_approx(s_row) : 0.f;
    // 8-bit codes: the planes 16 h and l of -q are not those of q negated, so the
    // signs go into the reciprocal (v * -rcp rounds as -v * rcp)
    wide_store_split<X, true>(a, v, row, block, lane, rcp, flip);
    return;
  }
  const float2 magic = make_float2(12582912.0f, 12582912.0f);
  float s_div = s_row;
  if (s_row > 0.f && s_row < 1.17549435e-38f) {
    s_div = s_row * kTwo64;
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __fmul2_rn(v[k], make_float2(kTwo64, kTwo64));
  }
  const float rcp = s_div > 0.f ? rcp_approx(s_div) : 0.f;
  const float2 rc2 = make_float2(rcp, rcp);
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = __ffma2_rn(v[k], rc2, magic);
  const float2 nmagic = make_float2(-12582912.0f, -12582912.0f);
  if constexpr (CODES == 1) {
    uint8_t* qrow = a.Q + static_cast<size_t>(row) * K + block;
#pragma unroll
    for (int c = 0; c < 4; ++c) {  // 16 codes a store
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = 8 * c + 2 * j;  // v[k], v[k + 1]: registers 2k .. 2k + 3
        uint16_t e0, e1;
        const float2 q0 = __fadd2_rn(v[k], nmagic), q1v = __fadd2_rn(v[k + 1], nmagic);
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(e0) : "f"(q0.y), "f"(q0.x));
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(e1) : "f"(q1v.y), "f"(q1v.x));
        w[j] = (static_cast<uint32_t>(e0) | (static_cast<uint32_t>(e1) << 16)) ^
               ((0u - ((flip >> (k >> 1)) & 1u)) & 0x80808080u);
      }
      *reinterpret_cast<uint4*>(qrow + wide_chunk<X>(c, lane)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  } else {
    // E2M3: 16 codes in 12 bytes (the packing of rq_device.cuh); runs of 64, 32
    // or 16 codes are 48, 24 or 12 bytes
    uint8_t* qrow = a.Q + static_cast<size_t>(row) * (3 * K / 4) + 3 * block / 4;
    constexpr int RUN = 4 >> X;  // consecutive chunks of 16 codes
#pragma unroll
    for (int c0 = 0; c0 < 4; c0 += RUN) {
      uint32_t o[3 * RUN];
#pragma unroll
      for (int c = 0; c < RUN; ++c) {  // a group of 16 codes -> 3 words
        uint32_t g[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int k = 8 * (c0 + c) + 2 * j;
          uint16_t e0, e1;
          const float2 q0 = __fadd2_rn(v[k], nmagic), q1v = __fadd2_rn(v[k + 1], nmagic);
          asm("cvt.rn.satfinite.e2m3x2.f32 %0, %1, %2;" : "=h"(e0) : "f"(q0.y), "f"(q0.x));
          asm("cvt.rn.satfinite.e2m3x2.f32 %0, %1, %2;" : "=h"(e1) : "f"(q1v.y), "f"(q1v.x));
          uint32_t w = static_cast<uint32_t>(e0) | (static_cast<uint32_t>(e1) << 16);
          w ^= (0u - ((flip >> (k >> 1)) & 1u)) & 0x20202020u;
          const uint32_t t = w - 3u * ((w >> 2) & 0x0FC00FC0u);
          g[j] = t - 15u * ((t >> 4) & 0x00FFF000u);
        }
        o[3 * c] = g[0] | (g[1] << 24);
        o[3 * c + 1] = (g[1] >> 8) | (g[2] << 16);
        o[3 * c + 2] = (g[2] >> 16) | (g[3] << 8);
      }
      uint8_t* q = qrow + 3 * wide_chunk<X>(c0, lane) / 4;
      if constexpr (RUN == 4) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          reinterpret_cast<uint4*>(q)[j] =
              make_uint4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
      } else if constexpr (RUN == 2) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          reinterpret_cast<uint2*>(q)[j] = make_uint2(o[2 * j], o[2 * j + 1]);
      } else {
#pragma unroll
        for (int j = 0; j < 3; ++j) reinterpret_cast<uint32_t*>(q)[j] = o[j];
      }
    }
  }
}

// Asymmetric codes of one row's 64-wide segment (Eq. 1 with the row's
// minimum and maximum as bounds, as in rq_device.cuh): delta = (max - min) /
// (2^n - 1) by the same division by a constant, q = rint((v - min) / delta) stored
// centered as q - 2^(n-1), 4 bits in E4M3 bytes (CODES 1) or 8 in split planes (2); kmax / kmin are the row's order keys of
// max and -min.  v holds the true transform (signs already restored).
template <int CODES, bool ROT, int X>
__device__ __forceinline__ void wide_quant_store_asym(const RotateQuantArgs& a, float2 (&v)[32],
                                                      int row, int seg, uint32_t kmax,
                                                      uint32_t kmin, int lane) {
  const int K = a.K;
  const int block = (seg >> X) << (6 + X);
  constexpr float div = CODES == 2 ? 255.0f : 15.0f;
  constexpr float rdiv = 1.0f / div;
  const float row_lo = -order_key_inv(kmin);
  const float am = __fsub_rn(order_key_inv(kmax), row_lo);
  const float q1 = am * rdiv;
  const float s_row = fmaf(fmaf(-div, q1, am), rdiv, q1);
  if (seg == 0) {
    a.S[row] = s_row;
    a.lo[row] = row_lo;
  }
  if (ROT) {
    float* dst = a.rot + static_cast<size_t>(row) * K + block;
#pragma unroll
    for (int q = 0; q < 16; ++q)
      *reinterpret_cast<float4*>(dst + wide_chunk<X>(q >> 2, lane) + 4 * (q & 3)) =
          make_float4(v[2 * q].x, v[2 * q].y, v[2 * q + 1].x, v[2 * q + 1].y);
  }
  // v <- rint((v - min) * (2^n - 1) / span) + 1.5 * 2^23 - 2^(n-1) (the centered
  // code in the low mantissa bits; 8 more for split planes); a constant row gets q
  // = 0; spans that asym_exact names take exact divisions.
  constexpr float mgc = CODES == 2 ? kSplitMagic - 128.0f : 12582912.0f - 8.0f;
  const float2 mg = make_float2(mgc, mgc);
  const float2 nlo = make_float2(-row_lo, -row_lo);
  if (asym_exact(am, div)) {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float2 d = __fadd2_rn(v[k], nlo);
      v[k] = __fadd2_rn(make_float2(__fmul_rn(__fdiv_rn(d.x, am), div),
                                    __fmul_rn(__fdiv_rn(d.y, am), div)),
                        mg);
    }
  } else {
    const float inv = am > 0.f ? div * rcp_approx(am) : 0.f;
    const float2 inv2 = make_float2(inv, inv);
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __ffma2_rn(__fadd2_rn(v[k], nlo), inv2, mg);
  }
  if constexpr (CODES == 2) {
    wide_store_split<X, false>(a, v, row, block, lane, 0.f, 0u);
    return;
  }
  const float2 nmagic = make_float2(-12582912.0f, -12582912.0f);
  uint8_t* qrow = a.Q + static_cast<size_t>(row) * K + block;
#pragma unroll
  for (int c = 0; c < 4; ++c) {  // 16 codes a store
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = 8 * c + 2 * j;
      uint16_t e0, e1;
      const float2 q0 = __fadd2_rn(v[k], nmagic), q1v = __fadd2_rn(v[k + 1], nmagic);
      asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(e0) : "f"(q0.y), "f"(q0.x));
      asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(e1) : "f"(q1v.y), "f"(q1v.x));
      w[j] = static_cast<uint32_t>(e0) | (static_cast<uint32_t>(e1) << 16);
    }
    *reinterpret_cast<uint4*>(qrow + wide_chunk<X>(c, lane)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// CODES 1 (E4M3), 2 (8-bit split planes) or 3 (E2M3); 64 <= b <= 256 (LOGB 6 ..
// 8); K % 64 == 0.  ASYM: asymmetric codes (a.lo != null), not E2M3.
// a.rows_per_tile = RH rows a tile (RH * 2K <= STAGE, RH * K / 64 <=
// blockDim.x).
template <typename T, int LOGB, int CODES, int STAGE, int STAGES, bool ROT, bool ASYM = false>
__global__ void __maxnreg__(kWideMaxRegs) rotate_quant_wide_kernel(RotateQuantArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  static_assert(LOGB >= 6 && LOGB <= 8, "wide loop: 64 <= b <= 256");
  static_assert(STAGE <= 65536, "gather offsets are 16-bit");
  static_assert(!ASYM || CODES != 3, "no asymmetric E2M3 codes");
  const int K = a.K;
  const int segs = K >> 6;
  const int RH = a.rows_per_tile;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const uint32_t row_bytes = static_cast<uint32_t>(K) * 2u;

  uint8_t* raw = smem;
  uint32_t* amax = reinterpret_cast<uint32_t*>(smem + STAGES * STAGE);  // [3][RH]
  uint32_t* amin = amax + 3 * RH;                                          // [3][RH]
  uint64_t* full = reinterpret_cast<uint64_t*>(
      (reinterpret_cast<uintptr_t>(amin + 3 * RH) + 7) & ~static_cast<uintptr_t>(7));
  int32_t* abort = reinterpret_cast<int32_t*>(full + STAGES);

  const int ntiles = (a.M + RH - 1) / RH;
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) mbar_init(&full[s], 1);
    *abort = 0;
    fence_mbarrier_init();
  }
  for (int i = tid; i < 6 * RH; i += blockDim.x) amax[i] = 0u;  // and amin
  __syncthreads();
  // This CTA's first tiles into L2 while the previous kernel drains; the
  // copies after the wait still read every value from L2 / memory, where the
  // previous kernel's writes land.
  if (tid == 0)
    for (int s = 0; s < STAGES; ++s) {
      const int t = static_cast<int>(blockIdx.x) + s * static_cast<int>(gridDim.x);
      if (t < ntiles) pair_prefetch<1>(a, RH, t);
    }
  const int items = RH * segs;
  const bool active = tid < items;
  const int r = active ? tid / segs : 0;
  const int seg = active ? tid - r * segs : 0;
  // XOR order: register pair k holds positions (2k) ^ m, (2k + 1) ^ m, m a
  // multiple of 8 below 64 that differs between neighbouring lanes (shared by
  // the lanes a cross-lane stage joins); the transform then comes out with
  // the sign (-1)^popc(i & m) on output i, constant over each 8 codes.
  const bool xor_order = (reinterpret_cast<uintptr_t>(a.perm) & 15u) == 0;
  const int xm = xor_order ? ((8 * (lane >> (LOGB - 6))) & 56) : 0;
  constexpr int X = LOGB - 6;  // butterfly stages across lanes
  const uint32_t flip = wide_flip<X>(xm, lane);
  // Gather offsets (bytes from the stage start) of positions (2k) ^ m and
  // (2k + 1) ^ m, low and high halves of ow[k].  An index outside [0, K) is
  // reported and replaced by column 0.
  uint32_t ow[32];
  {
    const uint32_t rbase = static_cast<uint32_t>(r) * row_bytes;
    const int32_t* pp = a.perm + seg * 64;
    bool bad = false;
    auto off = [&](int c) {
      const bool out = static_cast<unsigned>(c) >= static_cast<unsigned>(K);
      bad |= out;
      return rbase + 2u * static_cast<uint32_t>(out ? 0 : c);
    };
    if (xor_order) {
#pragma unroll
      for (int q = 0; q < 16; ++q) {  // positions 4q .. 4q + 3, read in the XOR order
        const int4 t = active ? __ldg(reinterpret_cast<const int4*>(pp) + (q ^ (xm >> 2)))
                              : make_int4(0, 0, 0, 0);
        ow[2 * q] = off(t.x) | (off(t.y) << 16);
        ow[2 * q + 1] = off(t.z) | (off(t.w) << 16);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const int c0 = active ? __ldg(pp + 2 * k) : 0;
        const int c1 = active ? __ldg(pp + 2 * k + 1) : 0;
        ow[k] = off(c0) | (off(c1) << 16);
      }
    }
    if (bad) record_status(a.status, CLQ_ERR_DEVICE_INDEX);
  }
  const uint32_t sbase = smem_addr(raw);
  const unsigned grp = __match_any_sync(0xffffffffu, active ? r : -1);
  const int leader = __ffs(grp) - 1;

  // X is read only from here on (the swap vector above is a layer constant; a
  // kernel of this library that writes one orders its writes before this grid).
  pdl_wait();
  pdl_launch_dependents();
  if (tid == 0)
    for (int s = 0; s < STAGES; ++s) {
      const int t = static_cast<int>(blockIdx.x) + s * static_cast<int>(gridDim.x);
      if (t < ntiles) pair_issue<STAGE, 1>(a, raw + s * STAGE, &full[s], RH, t);
    }

  bool done = false;
  for (int j0 = 0; !done; j0 += STAGES) {
#pragma unroll
    for (int s = 0; s < STAGES; ++s) {
      const int j = j0 + s;
      const int t = static_cast<int>(blockIdx.x) + j * static_cast<int>(gridDim.x);
      if (t >= ntiles) {
        done = true;
        break;
      }
      if (!pair_wait(&full[s], (j0 / STAGES) & 1, abort, a.status)) {
        done = true;
        if (tid == 0) {
          for (int s2 = 0; s2 < STAGES; ++s2)
            for (int ph = 0; ph < 2; ++ph)
              mbar_wait_bounded(&full[s2], ph, nullptr, nullptr, 10000000ull);
        }
        break;
      }
      const int row0 = RH * t;
      const int n = min(RH, a.M - row0);
      const int par = j % 3;

      // ---- 1. gather + first butterfly stage ------------------------------------
      float2 v[32];
      const uint32_t st = sbase + s * STAGE;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const uint16_t x0 = lds_u16(st + (ow[k] & 0xFFFFu));
        const uint16_t x1 = lds_u16(st + (ow[k] >> 16));
        v[k] = add_sub_mixed<T>(x0, to_f32<T>(x1));
      }
      // ---- 2. remaining stages, row maximum -----------------------------------
      wide_butterflies<LOGB>(v, lane);
      if constexpr (ASYM) {
        // the bounds are signed: restore each 4-code group's sign first
        if (X > 0 || xor_order) {
          uint32_t f = flip;
          asm volatile("" : "+r"(f));  // 16 factors kept over the loop would spill
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float sg = ((f >> q) & 1u) ? -1.f : 1.f;
            const float2 sg2 = make_float2(sg, sg);
            v[2 * q] = __fmul2_rn(v[2 * q], sg2);
            v[2 * q + 1] = __fmul2_rn(v[2 * q + 1], sg2);
          }
        }
        float mx, mn;
        wide_minmax(v, mx, mn);
        const unsigned kx = __reduce_max_sync(grp, order_key(mx));
        const unsigned kn = __reduce_max_sync(grp, order_key(-mn));
        if (active && lane == leader && r < n) {
          atomicMax(&amax[par * RH + r], kx);
          atomicMax(&amin[par * RH + r], kn);
        }
      } else {
        const unsigned kx = __reduce_max_sync(grp, __float_as_uint(wide_absmax(v)));
        if (active && lane == leader && r < n) atomicMax(&amax[par * RH + r], kx);
      }
      __syncthreads();  // row maxima complete; stage s fully read
      if (tid == 0) {
        const int t2 = t + STAGES * static_cast<int>(gridDim.x);
        if (t2 < ntiles) pair_issue<STAGE, 1>(a, raw + s * STAGE, &full[s], RH, t2);
      }
      // ---- 3. scale, codes, stores --------------------------------------------
      if (active && r < n) {
        if constexpr (ASYM)
          wide_quant_store_asym<CODES, ROT, X>(a, v, row0 + r, seg, amax[par * RH + r],
                                               amin[par * RH + r], lane);
        else
          wide_quant_store<CODES, ROT, X>(a, v, row0 + r, seg,
                                          __uint_as_float(amax[par * RH + r]), flip, lane);
      }
      if (tid < RH) {
        amax[((j + 2) % 3) * RH + tid] = 0u;
        if (ASYM) amin[((j + 2) % 3) * RH + tid] = 0u;
      }
    }
  }
  __syncthreads();
  if (tid == 0)
    for (int s = 0; s < STAGES; ++s) mbar_inval(&full[s]);
}

}  // namespace rq
}  // namespace clq
